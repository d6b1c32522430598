"""Host-side arithmetic of the cluster Cholesky (cluster_plan.cuh), compiled
with the host compiler.

* The failure words: rank 0 works one diagonal block ahead of the cluster's
  barriers, so a failed block's report must not be seen by a warp that still
  is to read the block before.  Every interleaving of rank 0 and one other warp
  over the panels' barriers is enumerated, with the word that the kernel uses.
* The row plans: a batch's shared memory is sized for its largest system, so no
  smaller system may need more.
"""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_04579_gb300", "csrc")
SHIM = r"""
#include "cluster_plan.cuh"
extern "C" {
int fail_word(int d) { return gnm::cl_fail_word(d); }
int plan(int n, int cs, int* out) { return gnm::cluster_plan(n, cs, out); }
long long fixed_doubles(int n) { return gnm::cl_fixed_doubles(n); }
int max_rows() { return gnm::kClMaxRows; }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cluster_plan")
    src, out = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(out)], check=True)
    so = ctypes.CDLL(str(out))
    so.fixed_doubles.restype = ctypes.c_longlong
    return so


def programs(attempts, nblk, word):
    """Rank 0's and another warp's operations over the attempts of one factor
    (attempts: the failing block of each, None for none), as in factor()."""
    w, r = [], []
    for a, bad in enumerate(attempts):
        r.append(("clear",))  # the words live in the reader's CTA, cleared ahead of the first barrier
        for prog in (w, r):
            prog.append(("arrive",))
            prog.append(("wait",))
        if bad == 0:
            w.append(("store", word(0)))
        for prog in (w, r):
            prog.append(("arrive",))
            prog.append(("wait",))
        w.append(("leave", bad == 0, a))
        r.append(("read", word(0), a, 0))
        for p in range(nblk - 1):
            for prog in (w, r):
                prog.append(("arrive",))
            if bad == p + 1:
                w.append(("store", word(p + 1)))
            for prog in (w, r):
                prog.append(("wait",))
                prog.append(("arrive",))
                prog.append(("wait",))
            w.append(("leave", bad == p + 1, a))
            r.append(("read", word(p + 1), a, p + 1))
        w.append(("end", a))
        r.append(("end", a))
    return w, r


def explore(attempts, nblk, word):
    """The set of blocks at which the reader left each attempt, over all
    interleavings (a stuck barrier counts as 'hang')."""
    w, r = programs(attempts, nblk, word)

    def after(prog, a):
        return next(i for i, op in enumerate(prog) if op[0] == "end" and op[1] == a) + 1

    seen, out, todo = set(), set(), [(0, 0, 0, 0, 0, 0, ())]
    while todo:
        s = todo.pop()
        if s in seen:
            continue
        seen.add(s)
        iw, ir, aw, ar, f0, f1, left = s
        moved = False
        for who in (0, 1):
            prog, i = (w, iw) if who == 0 else (r, ir)
            if i == len(prog):
                continue
            op = prog[i]
            n = [iw, ir, aw, ar, f0, f1, left]
            n[who] = i + 1
            if op[0] == "arrive":
                n[2 + who] += 1
            elif op[0] == "wait":
                if min(aw, ar) < n[2 + who]:
                    continue
            elif op[0] == "clear":
                n[4] = n[5] = 0
            elif op[0] == "store":
                n[4 + op[1]] = 1
            elif op[0] == "leave" and op[1]:
                n[0] = after(w, op[2])
            elif op[0] == "read" and (f0, f1)[op[1]]:
                n[6] = left + (op[3],)
                n[1] = after(r, op[2])
            elif op[0] == "end" and who == 1:
                n[6] = left + (None,)
            moved = True
            todo.append(tuple(n))
        if not moved:
            out.add(left if iw == len(w) and ir == len(r) else "hang")
    return out


@pytest.mark.parametrize("nblk", [1, 2, 3, 6])
def test_failed_blocks_are_seen_at_their_own_panel(lib, nblk):
    for first in range(nblk):
        for second in [None] + list(range(nblk)):
            assert explore([first, second], nblk, lib.fail_word) == {(first, second)}


def test_one_word_for_every_block_would_not_do():
    # the enumeration does see a report that arrives one panel early
    assert explore([2, None], 4, lambda d: 0) != {(2, None)}


@pytest.mark.parametrize("cs", [2, 3, 4, 5, 6, 7, 8, 10, 12, 14, 16])
def test_no_smaller_system_needs_more_than_the_largest(lib, cs):
    buf = (ctypes.c_int * 256)()
    worst = 0  # most shared memory over the smaller systems
    for nblk in range(1, 257):
        n = 16 * nblk
        most = lib.plan(n, cs, buf)
        if most >= 1 << 20:  # too many rows for a rank: such a cluster size is not taken
            break
        ranks = [buf[i] >> 24 for i in range(nblk)]
        assert max(ranks) < cs and max(ranks.count(q) for q in set(ranks)) <= lib.max_rows()
        # every row's blocks have a place of their own
        taken = set()
        for i in range(nblk):
            blocks = {(ranks[i], (buf[i] & 0xFFFFFF) + k) for k in range(i + 1)}
            assert not blocks & taken and max(b for _, b in blocks) < most
            taken |= blocks
        need = 8 * (lib.fixed_doubles(n) + 256 * most)
        assert need >= worst
        worst = need
