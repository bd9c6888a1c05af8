"""The eigCG window, vector by vector: Ritz values and residual norms of the grown basis.

Two comparisons.  Of the Ritz values that the vectors have (basis.ritz: H = U^H A U of what the window
held) with those of the projection T that the solver kept beside it (basis.pending): equal in exact
arithmetic, whatever the restarts kept.  And with the oracle, where its restarts kept all 2 nev columns
(where some are nearly dependent the rank is a matter of rounding, and of SVD there against Gram-Schmidt
here).

The solves are short (tol 1e-2 and 1e-3: 35 to 63 iterations, 0 to 30 restarts), so that rounding has not
yet spread through the Lanczos process: on the oracle a relative perturbation of 1e-15 in every product
moves these values by 5e-13 at most, one of 1e-7 by 5e-6.  A perturbation d of a Ritz vector moves its value
by up to d ||A||, and FP32 windows gather up to 1e-6 per restart, at random over 30 of them: bars of 1e-5
||A|| in FP32 and 1e-10 ||A|| in FP64.  A slot with the wrong vector moves a value by a good part of ||A||.
FP32 both inside the cluster and on the three launches of larger lattices.
"""
import numpy as np
import pytest

import oracle
from oracle import solvers
from paper_0707_0131_gb300 import _lib
from paper_0707_0131_gb300 import fixtures as fx

pytestmark = pytest.mark.gpu

M_Q = 0.05


@pytest.fixture(scope="module")
def api():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0707_0131_gb300 import api as a

    return a


def _cluster_launches(f):
    _lib.eig_profile_reset()
    _lib.eig_profile_enable(True)
    try:
        f()
    finally:
        _lib.eig_profile_enable(False)
    return sum(v["launches"] for n, v in _lib.eig_profile_read().items() if n == "cg_cluster")


@pytest.mark.parametrize("mode", ["fp64", "cluster", "launches"])
@pytest.mark.parametrize("dims", [(4, 6, 4, 8), (3, 5, 2, 7)])
def test_window_matches_the_oracle(api, monkeypatch, dims, mode):
    monkeypatch.setenv("EIG_CG_CLUSTER", "0" if mode == "launches" else "1")
    gauge = fx.make_gauge(dims, 83)
    W = oracle.Wilson(dims, M_Q, gauge)
    b = fx.make_rhs(dims, 84, 1).reshape(-1)
    norm = b
    for _ in range(60):
        norm = np.asarray(W.A(norm / np.linalg.norm(norm))).reshape(-1)
    bar = (1e-10 if mode == "fp64" else 1e-5) * np.linalg.norm(norm)
    # outputs of a restart (2 nev) at the edges of the FP64 restart's blocks, windows that fill up inside and
    # between blocks of 16 iterations, or not at all
    for nev, m, tol in [(1, 4, 1e-3), (2, 6, 1e-2), (5, 12, 1e-3), (8, 24, 1e-3), (9, 20, 1e-2), (10, 24, 1e-3),
                        (4, 40, 1e-3), (11, 24, 1e-2), (16, 34, 1e-3)]:
        kept = []
        o = solvers.eigcg(W, b, nev=nev, m=m, tol=tol, on_restart=lambda j, V, T, r: kept.append(V.shape[1]))
        op = api.Op(gauge, dims, M_Q, prec=64 if mode == "fp64" else 32)
        basis = api.Basis(op, 16)
        x = np.zeros_like(b)
        st = {}
        n = _cluster_launches(lambda: st.update(op.eigcg_solve(b, x, nev=nev, m=m, tol=tol, basis=basis)))
        assert (n > 0) == (mode == "cluster")
        pending = np.sort(basis.pending())
        basis.grow()
        th, rn = basis.ritz()
        order = np.argsort(th)
        th, rn = np.asarray(th)[order], np.asarray(rn)[order]
        assert len(th) == len(pending) and np.abs(th - pending).max() <= bar, (nev, m, th, pending)
        if all(c == 2 * nev for c in kept):
            V = o["V"]
            AV = np.stack([np.asarray(W.A(V[:, c])).reshape(-1) for c in range(V.shape[1])], axis=1)
            ref, S = np.linalg.eigh(V.conj().T @ AV)
            ref_rn = np.linalg.norm(AV @ S - (V @ S) * ref, axis=0)
            assert st["restarts"] == o["restarts"] and len(th) == len(ref), (nev, m)
            assert np.abs(th - ref).max() <= bar, (nev, m, th, ref)
            # a Ritz vector turns by the perturbation over its gap: its residual norm within 100 bars
            assert np.abs(rn - ref_rn).max() <= 100 * bar, (nev, m, rn, ref_rn)
        basis.close()
        op.close()


@pytest.mark.parametrize("max_iter", [1, 15, 37])
def test_iteration_limits_inside_a_block(api, monkeypatch, max_iter):
    """A limit that is not a multiple of the cluster's 16 iterations: as many iterations, and the same x, as
    with the three launches."""
    dims = (4, 6, 4, 8)
    gauge = fx.make_gauge(dims, 83)
    b = fx.make_rhs(dims, 84, 1).reshape(-1)
    xs = []
    for cluster in "10":
        monkeypatch.setenv("EIG_CG_CLUSTER", cluster)
        op = api.Op(gauge, dims, M_Q, prec=32)
        x = np.zeros_like(b)
        try:
            st = op.initcg_solve(b, x, tol=1e-12, max_iter=max_iter)[0]
            assert st["converged"] == 0 and st["iters"] == max_iter
        except _lib.EigError as e:
            assert "max_iter" in str(e)
        xs.append(x)
        op.close()
    # FP32 iterations from the same start: rounding of about 1e-7 per step
    assert np.linalg.norm(xs[0] - xs[1]) <= 1e-4 * np.linalg.norm(xs[1])


def test_fp64_restart_costs_its_outputs(api):
    """The FP64 window restart is bound by FP64 issue: 20 outputs cost 20 / 16 of 16 (they cost twice as much
    when the outputs were padded to 32)."""
    dims = (8, 8, 8, 8)
    op = api.Op(fx.make_gauge(dims, 85), dims, M_Q, prec=64)
    b = fx.make_rhs(dims, 86, 1).reshape(-1)
    ms = []
    for nev in (8, 10):
        best = np.inf
        for _ in range(3):
            _lib.eig_profile_reset()
            _lib.eig_profile_enable(True)
            op.eigcg_solve(b, np.zeros_like(b), nev=nev, m=100, tol=1e-9)
            _lib.eig_profile_enable(False)
            r = _lib.eig_profile_read()["window_restart"]
            best = min(best, r["ms"] / r["launches"])
        ms.append(best)
    op.close()
    assert ms[1] <= 1.5 * ms[0], ms
