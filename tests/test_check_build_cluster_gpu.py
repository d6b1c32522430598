"""The bounds-check build on the cluster Cholesky: its stores to its own and
the other ranks' shared memory and to the system's copy are checked, none is
out of range, and the results are the normal build's bit for bit -- with the
largest cluster, two CTAs per instance, uneven systems (down to one panel) and
factorisations that fail and are retried."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASES = r"""
import json, sys
import numpy as np
sys.path.insert(0, sys.argv[2])
from paper_2512_04579_gb300 import gnmppi as G
from paper_2512_04579_gb300 import inputs as I
G.load(sys.argv[1])
out, ctas = {}, {}
def case(name, prob, batch, x0, tgt, n, shapes=None):
    s = G.Solver(prob, batch, shapes)
    st, U, rep = s.step(x0, tgt, np.full(n, 0.01), np.full(n, 0.2), 0)
    out[name] = [U.ravel().tolist(), [[r.status, r.chol_retries, r.step_norm] for r in rep]]
    ctas[name] = G.gnmppi_tune_report(s.h)["solve_ctas"]
    s.close()
for name, N, b, prec in (("n34", 17, 1, G.PREC_FP64), ("n200", 100, 1, G.PREC_BF16), ("n200x70", 100, 70, G.PREC_FP32),
                         ("n400", 200, 1, G.PREC_BF16), ("n640", 320, 1, G.PREC_BF16)):
    x0, tgt = I.chain_instances(11 + N, b, 4)
    case(name, G.chain_problem(4, N=N, K=4 * N + 64, precision=prec, sigma0=0.2, seed=5), b, x0, tgt, 2 * N * b)
shapes = [(8 * b + 5, 3, 256) for b in range(6)]
x0 = np.concatenate([I.chain_instances(b, 1, 3)[0].ravel() for b in range(6)])
tgt = np.concatenate([I.chain_instances(b, 1, 3)[1].ravel() for b in range(6)])
case("uneven", G.chain_problem(3, N=30, K=256, precision=G.PREC_FP32, sigma0=0.2, seed=6), 6, x0, tgt,
     sum(2 * s[0] for s in shapes), shapes)
x0, tgt = I.chain_instances(4, 8, 10)
case("retried", G.chain_problem(10, N=100, K=400, precision=G.PREC_BF16, sigma0=0.2, seed=9, lam=1e-9), 8, x0, tgt, 1600)
print(json.dumps({"out": out, "ctas": ctas, "offences": int(G.load().gnmppi_check_count())}))
"""


def _run(lib_path):
    r = subprocess.run([sys.executable, "-c", CASES, lib_path, ROOT], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_check_build_counts_no_offence_on_clusters():
    from paper_2512_04579_gb300 import build as B

    normal = _run(B.build())
    checked = _run(B.build(check=True))
    assert min(normal["ctas"].values()) >= 2 and checked["ctas"] == normal["ctas"]
    assert normal["offences"] == -1 and checked["offences"] == 0
    assert checked["out"] == normal["out"]
