"""The fixed-point form of the FP64 stencil is optional: an operator takes it when there is room, gives it
back to any allocation of its own that finds none, and takes it again with the next workspace.

EIG_TEST_ALLOC_LIMIT fakes a device without room for larger requests, EIG_TEST_ALLOC_TOTAL one that
holds so many bytes in all.
"""
import numpy as np
import pytest

import oracle
from paper_0707_0131_gb300 import _lib
from paper_0707_0131_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu

DIMS = (7, 9, 15, 31)  # odd number of sites: the fixed-point field is larger than the natural one


@pytest.fixture(scope="module")
def api():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0707_0131_gb300 import api as a

    return a


@pytest.mark.parametrize("prec,which", [(64, 2), (32, 3)])
def test_comes_back_after_a_tight_moment(api, monkeypatch, prec, which):
    gauge = fx.make_gauge(DIMS, 71)
    op = api.Op(gauge, DIMS, -0.1, prec=prec)
    psi = fx.make_rhs(DIMS, 72, 1).reshape(-1)
    first, tight, again = np.empty_like(psi), np.empty_like(psi), np.empty_like(psi)
    op.apply(which, psi, first)
    full = op.trim()
    monkeypatch.setenv("EIG_TEST_ALLOC_LIMIT", str(op.V * 192))
    op.apply(which, psi, tight)
    assert op.trim() < full and not np.array_equal(tight, first)  # the FP64 stencil's rounding
    monkeypatch.delenv("EIG_TEST_ALLOC_LIMIT")
    op.apply(which, psi, again)
    assert np.array_equal(again, first) and op.trim() == full
    op.close()


def _work(api, gauge, psi):
    """One operator with a basis through products and solves; its results."""
    op = api.Op(gauge, DIMS, 0.3, prec=64)
    basis = None
    try:
        basis = api.Basis(op, 8)
        out, x = np.empty_like(psi), np.zeros_like(psi)
        op.apply(2, psi, out)
        st = op.eigcg_solve(psi, x, nev=4, m=12, tol=1e-8, basis=basis)
        basis.grow()
        y = np.zeros_like(psi)
        op.trim()
        sts = op.initcg_solve(psi, y, tol=1e-8, basis=basis)
        return out, x, y, st, sts[0]
    finally:
        if basis is not None:
            basis.close()
        op.close()


def test_fits_wherever_the_fp64_stencil_fits(api, monkeypatch):
    """The smallest device that an operator whose links do not suit the fixed-point form works on is
    enough for one that would like it too."""
    gauge = fx.make_gauge(DIMS, 73)
    psi = fx.make_rhs(DIMS, 74, 1).reshape(-1)
    uneven = gauge.copy()
    uneven[0, 0] *= 0.01

    def fits(total):
        monkeypatch.setenv("EIG_TEST_ALLOC_TOTAL", str(total))
        try:
            _work(api, uneven, psi)
            return True
        except _lib.EigError as e:
            assert e.status == _lib.EIG_ERR_OOM
            return False

    lo, hi = 0, 2 << 30
    assert fits(hi)
    while hi - lo > 1 << 20:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid) else (mid, hi)
    monkeypatch.setenv("EIG_TEST_ALLOC_TOTAL", str(hi))
    out, x, y, st, st2 = _work(api, gauge, psi)
    W = oracle.Wilson(DIMS, 0.3, gauge)
    ref = np.asarray(W.A(psi)).reshape(-1)
    assert np.linalg.norm(out - ref) <= 1e-14 * np.linalg.norm(ref)
    for v, s in ((x, st), (y, st2)):
        assert s["converged"] == 1
        assert np.linalg.norm(psi - np.asarray(W.A(v)).reshape(-1)) <= 1e-8 * np.linalg.norm(psi)
