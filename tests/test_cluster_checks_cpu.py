"""Every store of the cluster Cholesky to shared or global memory is one that
the bounds-check build tests: a store through a subscript or a pointer in
chol_cluster.cuh stands behind has() or GNM_IN()."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_04579_gb300", "csrc")
# arrays that are registers, flags of fixed size, and the words behind the columns that has() covers
LOCAL = re.compile(r"^(h|l|x|y|cur|nxt|acc|fail|col)\[|^\*cl_map\(fail")


def test_stores_are_checked():
    lines = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "chol_cluster.cuh")).read()).split("\n")
    store = re.compile(r"(?:^|\) |\) \{ |; )((?:\*?[\w.:<>]+(?:\([^=;]*\))?(?:\[[^=;]*\])*)|\*[\w]+) [-+]?= ")
    unchecked = []
    for k, line in enumerate(lines):
        m = store.search(line.strip())
        if not m or ("[" not in m.group(1) and not m.group(1).startswith("*")):
            continue
        target = m.group(1).lstrip()
        if LOCAL.match(target):
            continue
        if not re.search(r"has\(|GNM_IN\(", "\n".join(lines[max(0, k - 5) : k + 1])):
            unchecked.append((k + 1, line.strip()))
    assert not unchecked, unchecked
