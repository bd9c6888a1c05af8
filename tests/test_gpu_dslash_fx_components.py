"""The fixed-point FP64 stencil component by component: fields whose components, spins, colours or sites
differ by many orders of magnitude, point sources and fields near the ends of the exponent range.

The same vectors alone (FP64 arithmetic) and two together (fixed point with FP64 where its guard asks
for it).  A component's bound is relative to the sum of its own terms |u_ab| |h_b|, as fxmath.h derives
it: 61 of 2^-53 for a kept element's hop sum and 16 for the FP64 chain's (a +- b, six products, eight
hops), halved by the factor of the hop term, and four for the centre term and the last sum.
"""
import numpy as np
import pytest

from paper_0707_0131_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu

U53 = 2.0 ** -53


@pytest.fixture(scope="module")
def api():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0707_0131_gb300 import api as a

    return a


def _hop_terms(gauge, dims, psi, dagger):
    """Sum over the hops of |U| |psi_s -+ B_mu psi_partner| per output component (psi [k, V, 4, 3])."""
    lx, ly, lz, lt = dims
    f = psi.reshape(-1, lt, lz, ly, lx, 4, 3)
    u = np.abs(np.asarray(gauge)).reshape(lt, lz, ly, lx, 4, 3, 3)
    out = np.zeros(f.shape)
    part = [(1, 0), (1, 0), (0, 1), (0, 1)]
    fac = [(1j, 1j), (-1, 1), (1j, -1j), (1, 1)]
    for mu in range(4):
        for back in (False, True):
            sg = (1 if back else -1) * (-1 if dagger else 1)
            g = f if back else np.roll(f, -1, axis=4 - mu)
            h = np.stack([np.abs(g[..., s, :] + sg * fac[mu][s] * g[..., 2 + part[mu][s], :]) for s in (0, 1)], axis=-2)
            um = u[..., mu, :, :]
            w = np.einsum("tzyxba,ktzyxsb->ktzyxsa" if back else "tzyxab,ktzyxsb->ktzyxsa", um, h)
            if back:
                w = np.roll(w, 1, axis=4 - mu)
            out[..., :2, :] += w
            for s in (0, 1):
                out[..., 2 + s, :] += w[..., part[mu][s], :]
    return out.reshape(psi.shape)


def _field(rng, kind, shape):
    v = rng.normal(size=shape) + 1j * rng.normal(size=shape)
    if kind == "colours":
        v *= [1.0, 1e-9, 1e-18]
    elif kind == "spins":
        v *= np.array([1e-12, 1.0, 1e-9, 1e-12])[:, None]
    elif kind == "sites":
        v *= 10.0 ** -rng.uniform(0, 12, size=(*shape[:2], 1, 1))
    elif kind == "components":
        v *= 10.0 ** -rng.uniform(0, 6, size=shape)
    elif kind == "point":
        keep = v[:, 1234, 1, 2].copy()
        v[:] = 0
        v[:, 1234, 1, 2] = keep
    elif kind == "one spin":
        v[:, :, 1:] = 0
    elif kind == "subnormal":
        v *= 3e-310
    return v


@pytest.mark.parametrize("links", ["random", "unit"])
@pytest.mark.parametrize("kind", ["colours", "spins", "sites", "components", "point", "one spin", "subnormal"])
def test_products_hold_every_component(api, links, kind):
    dims, m_q = (8, 8, 8, 8), 0.05
    gauge = fx.make_gauge(dims, 91)
    if links == "unit":
        gauge = np.zeros_like(gauge)
        gauge[...] = np.eye(3).reshape((1,) * (gauge.ndim - 2) + (3, 3))
    op = api.Op(gauge, dims, m_q, prec=64, max_rhs=2)
    psi = _field(np.random.default_rng(92), kind, (2, op.V, 4, 3))
    for which in (0, 1):
        one, two = np.empty_like(psi), np.empty_like(psi)
        for r in range(2):
            op.apply(which, np.ascontiguousarray(psi[r:r + 1]), one[r:r + 1], 1)
        op.apply(which, psi, two, 2)
        terms = _hop_terms(gauge, dims, psi, which == 1)
        bar = U53 * (39 * terms + 4 * (4 + m_q) * np.abs(psi)) + 64 * 2.0 ** -1074
        err = np.abs(two - one)
        assert np.all(err <= bar), (which, (err / np.maximum(bar, 1e-320)).max())
        assert kind not in ("subnormal",) or np.abs(two - (4 + m_q) * psi).max() > 0  # the hop sum is there
    op.close()


@pytest.mark.parametrize("even_odd", [False, True])
@pytest.mark.parametrize("prec", [64, 32])
def test_colours_of_unit_links_stay_apart(api, even_odd, prec):
    """Products and solves where only colour 0 has a source: the others stay exactly zero, in every
    epilogue (FP64 operators iterate on the fixed-point stencil, mixed ones take residuals from it)."""
    dims = (8, 8, 8, 8)
    k = 4 if even_odd else 2  # 8192 pairs
    gauge = np.zeros_like(fx.make_gauge(dims, 93))
    gauge[...] = np.eye(3).reshape((1,) * (gauge.ndim - 2) + (3, 3))
    op = api.Op(gauge, dims, 0.4, prec=prec, max_rhs=k, even_odd=even_odd)
    rng = np.random.default_rng(94)
    b = np.zeros((k, op.V, 4, 3), dtype=complex)
    for r in range(k):
        b[r, rng.integers(op.V), rng.integers(4), 0] = 1.0
    x = np.zeros_like(b)
    st = op.initcg_solve(b, x, tol=1e-10, k=k)
    assert all(s["converged"] == 1 for s in st)
    assert np.abs(x[..., 0]).max() > 0 and np.all(x[..., 1:] == 0)
    if prec == 64:
        psi = rng.normal(size=(k, op.Vf, 4, 3)) * np.array([1.0, 1e-20, 0.0]) + 0j
        one, two = np.empty_like(psi), np.empty_like(psi)
        for r in range(k):
            op.apply(2, np.ascontiguousarray(psi[r:r + 1]), one[r:r + 1], 1)
        op.apply(2, psi, two, k)
        # four chains of hops (two per M of the odd-even form), each bounded as above with sums of terms
        # below 16 sites' spinors: 4 * 60 * 16 of 2^-53 of the colour's largest component times a few
        bar = 2.0 ** -53 * 8e3 * np.abs(psi).max(axis=(1, 2))[:, None, None, :] * 8
        assert np.all(np.abs(two - one) <= bar)
        assert np.all(two[..., 2] == 0)
    op.close()


@pytest.mark.parametrize("sizes", [(3.0, 3.0, 3.0, 3.0), (0.06, 0.06, 0.06, 0.06), (1.0, 0.5, 1.2, 0.2), (1e30, 1e30, 1e30, 1e29)])
def test_links_of_other_sizes(api, sizes):
    """Links that are not unitary (smeared, anisotropic): the bound of unit rows times sqrt 2 for the
    power of two they are held relative to, as above, (61 sqrt 2 + 16) / 2 < 52."""
    dims, m_q = (8, 8, 8, 8), 0.05
    gauge = fx.make_gauge(dims, 95) * np.array(sizes)[:, None, None]
    op = api.Op(gauge, dims, m_q, prec=64, max_rhs=2)
    psi = _field(np.random.default_rng(96), "gauss", (2, op.V, 4, 3))
    for which in (0, 1):
        one, two = np.empty_like(psi), np.empty_like(psi)
        for r in range(2):
            op.apply(which, np.ascontiguousarray(psi[r:r + 1]), one[r:r + 1], 1)
        op.apply(which, psi, two, 2)
        bar = U53 * (52 * _hop_terms(gauge, dims, psi, which == 1) + 4 * (4 + m_q) * np.abs(psi))
        assert np.all(np.abs(two - one) <= bar), which
    op.close()


def test_links_of_other_sizes_are_as_fast(api):
    """The residuals' product of a mixed operator costs the same whatever the size of the links (it took
    twice as long where they were left to the FP64 stencil)."""
    import time

    import torch

    dims = (12, 12, 12, 24)
    best = []
    for size in (1.0, 3.0):
        op = api.Op(size * fx.make_gauge(dims, 97), dims, 0.05, prec=32)
        x = torch.randn(op.V * 12, dtype=torch.complex128, device="cuda")
        y = torch.empty_like(x)
        t = []
        for _ in range(30):
            t0 = time.perf_counter()
            op.apply(3, x, y)
            t.append(time.perf_counter() - t0)
        best.append(min(t))
        op.close()
    assert best[1] <= 1.4 * best[0], best


@pytest.mark.parametrize("dims,k", [((7, 9, 7, 21), 1), ((8, 8, 8, 20), 1), ((7, 9, 7, 12), 2)])
def test_device_vectors_on_both_sides_of_the_natural_rule(api, dims, k):
    """Device vectors of 8192 to 10239 pairs are read and written where they are, host vectors and larger
    device ones go through the fixed-point form: the same products (bounds of the components test)."""
    import torch

    m_q = 0.05
    gauge = fx.make_gauge(dims, 98)
    op = api.Op(gauge, dims, m_q, prec=64, max_rhs=k)
    psi = _field(np.random.default_rng(99), "gauss", (k, op.V, 4, 3))
    for which in (0, 1):
        host = np.empty_like(psi)
        op.apply(which, psi, host, k)
        vin = torch.from_numpy(psi).cuda()
        vout = torch.empty_like(vin)
        op.apply(which, vin, vout, k)
        bar = U53 * (39 * _hop_terms(gauge, dims, psi, which == 1) + 4 * (4 + m_q) * np.abs(psi))
        assert np.all(np.abs(vout.cpu().numpy() - host) <= bar), which
    op.close()
