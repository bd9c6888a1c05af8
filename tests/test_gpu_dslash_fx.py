"""The fixed-point FP64 stencil (launches of at least 8192 (site, RHS) pairs, unitary links).

Each neighbour enters with at most 2^-55 of the largest component of the eight (alignment and limb
truncation), so on Gaussian vectors (largest of ~200 components about 4.5 standard deviations,
outputs about 8) the error stays below 8 * 2^-55 * 4.5 / 8 plus one rounding: under 1e-15 of the
norm.  Launches below the threshold run the FP64 arithmetic, which the k = 1 calls use here.
"""
import numpy as np
import pytest

import oracle
from oracle import wilson_eo
from paper_0707_0131_gb300 import _lib
from paper_0707_0131_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0707_0131_gb300 import api as a

    return a


def _rel(out, ref):
    return np.linalg.norm(out - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("dims,k", [((7, 9, 7, 21), 1), ((2, 3, 64, 22), 1), ((8, 8, 8, 8), 2), ((5, 6, 7, 5), 16)])
def test_products(api, dims, k):
    gauge = fx.make_gauge(dims, 71)
    W = oracle.Wilson(dims, -0.1, gauge)
    op = api.Op(gauge, dims, -0.1, prec=64, max_rhs=k)
    psi = fx.make_rhs(dims, 72, k).reshape(k, -1)
    assert psi.shape[1] // 12 * k >= 8192
    for which, f in [(0, W.M), (1, W.Mdag), (2, W.A)]:
        out = np.empty_like(psi)
        op.apply(which, psi, out, k)
        for r in range(k):
            assert _rel(out[r], np.asarray(f(psi[r])).reshape(-1)) < 1e-15, (which, r)
    op.close()
    # the same through a mixed-precision operator (its FP64 products)
    op = api.Op(gauge, dims, -0.1, prec=32, max_rhs=k)
    out = np.empty_like(psi)
    op.apply(3, psi, out, k)
    for r in range(k):
        assert _rel(out[r], np.asarray(W.A(psi[r])).reshape(-1)) < 1e-15
    op.close()


def test_odd_even(api):
    dims, k = (8, 8, 8, 8), 4
    gauge = fx.make_gauge(dims, 73)
    W = wilson_eo.WilsonEO(dims, 0.05, gauge)
    op = api.Op(gauge, dims, 0.05, prec=64, max_rhs=k, even_odd=True)
    psi = np.ascontiguousarray(fx.make_rhs(dims, 74, k).reshape(k, -1)[:, : W.N])
    for which, f in [(0, W.Mhat), (1, W.Mhat_dag), (2, W.A)]:
        out = np.empty_like(psi)
        op.apply(which, psi, out, k)
        for r in range(k):
            assert _rel(out[r], np.asarray(f(psi[r])).reshape(-1)) < 1e-15, (which, r)
    op.close()


@pytest.mark.parametrize("kind", ["point", "graded", "huge", "tiny", "zero", "nan", "inf"])
def test_against_fp64_path(api, kind):
    """Vectors far from uniform: two RHS together (fixed point) against each alone (FP64 arithmetic)."""
    dims = (8, 8, 8, 8)
    gauge = fx.make_gauge(dims, 75)
    op = api.Op(gauge, dims, 0.05, prec=64, max_rhs=2)
    psi = fx.make_rhs(dims, 76, 2).reshape(2, -1, 12)
    if kind == "point":
        keep = psi[:, 1234, 5].copy()
        psi[:] = 0
        psi[:, 1234, 5] = keep
    elif kind == "graded":
        psi *= 10.0 ** (-np.arange(psi.shape[1]) % 37)[None, :, None]
    elif kind == "huge":
        psi *= 1e300
    elif kind == "tiny":
        psi *= 1e-290
    elif kind == "zero":
        psi[:] = 0
    else:
        psi[1, 777, 3] = np.nan if kind == "nan" else np.inf
    psi = psi.reshape(2, -1)
    for which in (0, 1, 2):
        one, two = np.empty_like(psi), np.empty_like(psi)
        for r in range(2):
            op.apply(which, np.ascontiguousarray(psi[r:r + 1]), one[r:r + 1], 1)
        op.apply(which, psi, two, 2)
        a, b = one.view(np.float64), two.view(np.float64)
        assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
        ok = np.isfinite(a)
        # site by site, against the largest component that reaches the site
        scale = np.zeros((2, *dims[::-1]))
        mag = np.where(np.isfinite(psi), np.abs(psi), 0).reshape(2, *dims[::-1], 12).max(-1)
        for step in range(2 if which == 2 else 1):
            scale = mag.copy()
            for ax in range(1, 5):
                scale = np.maximum(scale, np.maximum(np.roll(mag, 1, ax), np.roll(mag, -1, ax)))
            mag = scale
        err = np.where(ok, np.abs(np.where(ok, a, 0) - np.where(ok, b, 0)), 0).reshape(2, *dims[::-1], 24).max(-1)
        assert np.all(err <= 64 * 2.0 ** -52 * scale * (70 if which == 2 else 1)), (which, (err / np.maximum(scale, 1e-300)).max())
    op.close()


def test_links_that_are_not_unitary_keep_fp64(api):
    dims, k = (8, 8, 8, 8), 2
    gauge = 3.0 * fx.make_gauge(dims, 77)
    W = oracle.Wilson(dims, 0.05, gauge)
    op = api.Op(gauge, dims, 0.05, prec=64, max_rhs=k)
    psi = fx.make_rhs(dims, 78, k).reshape(k, -1)
    out = np.empty_like(psi)
    op.apply(0, psi, out, k)
    for r in range(k):
        assert _rel(out[r], np.asarray(W.M(psi[r])).reshape(-1)) < 1e-12
    op.close()


@pytest.mark.parametrize("when", ["links", "workspace"])
def test_no_room_for_the_fixed_point_form(api, monkeypatch, when):
    """An allocation limit that fits the FP64 links and fields but not their fixed-point forms
    (rounded up to 32 elements): the operator works with the FP64 stencil."""
    dims = (7, 9, 15, 31)  # the links larger than the 16 MB of reduction scratch
    V = int(np.prod(dims))
    assert V % 32
    gauge = fx.make_gauge(dims, 71)
    W = oracle.Wilson(dims, -0.1, gauge)
    psi = fx.make_rhs(dims, 72, 1).reshape(-1)
    op = api.Op(gauge, dims, -0.1, prec=64, max_rhs=1)
    full = _lib.eig_op_trim(op.h)
    if when == "links":
        op.close()
        monkeypatch.setenv("EIG_TEST_ALLOC_LIMIT", str(V * 576))
        op = api.Op(gauge, dims, -0.1, prec=64, max_rhs=1)
    else:
        monkeypatch.setenv("EIG_TEST_ALLOC_LIMIT", str(V * 192))
    out = np.empty_like(psi)
    op.apply(2, psi, out, 1)
    assert _rel(out, np.asarray(W.A(psi)).reshape(-1)) < 1e-15
    assert _lib.eig_op_trim(op.h) < full  # no exponents, no rounding of the field
    op.close()
