"""CG iterations inside one thread-block cluster (FP32, at most 4096 (site, RHS) pairs).

Edges: extents of 2 and odd extents, fewer pairs than threads, a ragged last CTA, every batch width,
both link formats (forced), the largest size and the first beyond it; eigCG windows that fill up and
restart inside and between blocks of iterations.  Bars: those of the solver tests (true residual as the
oracle recomputes it within tol, iterations within 10% of the oracle's).
"""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import numpy as np, oracle
from oracle import solvers
from paper_0707_0131_gb300 import api, fixtures as fx
for dims, k in [((2, 2, 2, 2), 1), ((3, 2, 5, 2), 2), ((5, 3, 7, 3), 1), ((4, 4, 4, 4), 16), ((6, 4, 2, 10), 8),
                ((8, 8, 8, 8), 1), ((3, 5, 7, 39), 1), ((7, 9, 5, 13), 1)]:
    gauge = fx.make_gauge(dims, 81)
    W = oracle.Wilson(dims, 0.2, gauge)
    op = api.Op(gauge, dims, 0.2, prec=32, max_rhs=k)
    B = fx.make_rhs(dims, 82, k).reshape(k, -1)
    X = np.zeros_like(B)
    st = op.initcg_solve(B, X, tol=1e-9, k=k)
    for r in range(k):
        res = np.linalg.norm(B[r] - np.asarray(W.A(X[r])).reshape(-1)) / np.linalg.norm(B[r])
        assert st[r]["converged"] == 1 and res <= 1e-9, (dims, k, r, st[r], res)
        o = solvers.cg(W, B[r], tol=1e-9)
        assert abs(st[r]["iters"] - o["iters"]) <= max(2, 0.1 * o["iters"]), (dims, k, r, st[r]["iters"], o["iters"])
    op.close()
dims = (4, 6, 4, 8)
gauge = fx.make_gauge(dims, 83)
W = oracle.Wilson(dims, 0.05, gauge)
b = fx.make_rhs(dims, 84, 1).reshape(-1)
for nev, m in [(2, 6), (8, 24), (4, 40)]:
    op = api.Op(gauge, dims, 0.05, prec=32)
    basis = api.Basis(op, 16)
    x = np.zeros_like(b)
    st = op.eigcg_solve(b, x, nev=nev, m=m, tol=1e-8, basis=basis)
    assert np.linalg.norm(b - np.asarray(W.A(x)).reshape(-1)) / np.linalg.norm(b) <= 1e-8
    o = solvers.eigcg(W, b, nev=nev, m=m, tol=1e-8)
    assert abs(st["iters"] - o["iters"]) <= max(2, 0.1 * o["iters"]), (nev, m, st["iters"], o["iters"])
    basis.grow()
    th, rn = basis.ritz()
    lam = np.min(th)
    assert np.all(th > 0) and rn[0] < 0.2 * 66, (nev, m, th, rn)
    U = basis.vectors()
    assert np.linalg.norm(U.conj().T @ U - np.eye(U.shape[1])) < 1e-5
    basis.close()
    op.close()
print("cluster ok")
"""


@pytest.mark.parametrize("links", ["12", "18"])
def test_cluster_solves(links):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, "-c", CHILD], env=dict(os.environ, EIG_DSLASH_LINKS=links), cwd=root,
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0 and "cluster ok" in p.stdout, p.stdout[-2000:] + p.stderr[-4000:]
