"""The stencil that spreads a site's hops over lanes (small lattices) against the oracle.

Sizes at its edges: extents of 2 and odd extents, fewer (site, RHS) pairs than one block, a ragged
last block, several passes per block, every batch width's RHS-to-group mapping.  FP64 device vectors
are read and written in the natural layout, so disjoint, identical and overlapping in / out are all
tried.  Bars: those of test_gpu_dslash.py (1e-12 in FP64).
"""
import numpy as np
import pytest

import oracle
from paper_0707_0131_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0707_0131_gb300 import api as a

    return a


@pytest.mark.parametrize("dims,k", [((2, 2, 2, 2), 1), ((3, 2, 5, 2), 2), ((4, 4, 4, 4), 1), ((6, 4, 2, 10), 16),
                                    ((5, 7, 3, 9), 4), ((8, 8, 8, 8), 1), ((8, 8, 8, 8), 4)])
def test_fp64_device_vectors(api, dims, k):
    import torch

    gauge = fx.make_gauge(dims, 61)
    W = oracle.Wilson(dims, -0.1, gauge)
    op = api.Op(gauge, dims, -0.1, prec=64, max_rhs=k)
    psi = fx.make_rhs(dims, 62, k).reshape(k, -1)
    n = psi.size
    for which, f in [(0, W.M), (1, W.Mdag), (2, W.A)]:
        ref = np.stack([np.asarray(f(psi[r])).reshape(-1) for r in range(k)])
        # apart, in place, and out one site behind in within one buffer
        for gap in (n, 0, 12):
            buf = torch.zeros(2 * n + 12, dtype=torch.complex128, device="cuda")
            vin, vout = buf[gap:gap + n], buf[:n]
            vin.copy_(torch.from_numpy(psi.reshape(-1)))
            op.apply(which, vin, vout, k)
            out = vout.cpu().numpy().reshape(k, -1)
            err = np.linalg.norm(out - ref, axis=1) / np.linalg.norm(ref, axis=1)
            assert err.max() < 1e-12, (which, gap, err)
    op.close()


@pytest.mark.parametrize("dims,k", [((2, 2, 2, 2), 1), ((4, 4, 4, 4), 2), ((6, 4, 2, 10), 8)])
def test_fp64_solve_epilogues(api, dims, k):
    """The norm, CG and residual epilogues: a batch reaches 1e-10, each residual as the oracle recomputes it."""
    gauge = fx.make_gauge(dims, 63)
    W = oracle.Wilson(dims, 0.3, gauge)
    op = api.Op(gauge, dims, 0.3, prec=64, max_rhs=k)
    B = fx.make_rhs(dims, 64, k).reshape(k, -1)
    X = np.zeros_like(B)
    st = op.initcg_solve(B, X, tol=1e-10, k=k)
    for r in range(k):
        res = np.linalg.norm(B[r] - np.asarray(W.A(X[r])).reshape(-1)) / np.linalg.norm(B[r])
        assert st[r]["converged"] == 1 and res <= 1e-10, (r, st[r], res)
    op.close()
