// Internal header: the epilogues of the stencils and the scalar updates that follow their
// reductions, shared by the one-thread, split, fixed-point and cluster kernels.
#pragma once
#include "kernels.cuh"

namespace eig {

// epilogues: the numbers of dslash.cu's Epi and dslash32.cuh's E_*
enum { SPL_PLAIN = 0, SPL_NORM = 1, SPL_CG = 2, SPL_RESID = 3 };

namespace {

// the scalar updates of RHS r after a grid reduction gave tot (Fig. 1 steps 12, 4, 8; see
// kernels.cuh for the launches they belong to)
template <int EPI>
__device__ __forceinline__ void finish_scalars(CGScalars *sts, double *h_alpha, double *h_beta, double *h_rho, int iter,
                                               int k, int set_rho, int r, double tot) {
    CGScalars &st = sts[r];
    const long hi = (long)iter * k + r;
    if (EPI == SPL_NORM) {
        if (st.active) {
            st.pAp = tot;
            if (!(tot > 0.0) || !isfinite(tot)) {
                st.breakdown = 1;
                st.active = 0;
                st.alpha = 0.0;
            } else {
                st.alpha = st.rho / tot;
            }
            h_alpha[hi] = st.alpha;
            st.x_pending = st.active;
        } else {
            st.alpha = 0.0;
            st.x_pending = 0;
        }
    } else if (EPI == SPL_CG) {
        if (st.active) {
            if (!isfinite(tot)) {
                st.breakdown = 1;
                st.active = 0;
                return;
            }
            st.iters = iter;
            st.nit++;
            st.rho_prev = st.rho;
            st.rho = tot;
            st.beta = tot / st.rho_prev;
            h_rho[hi] = tot;
            h_beta[hi + k] = st.beta;
            if (tot <= st.target) st.active = 0;
        }
    } else if (EPI == SPL_RESID) {
        st.aux = tot;
        if (set_rho) {
            st.rho = tot;
            st.beta = tot / st.rho_prev;
            h_rho[hi] = tot;
            h_beta[hi + k] = st.beta;
        }
    }
}

}  // namespace
}  // namespace eig
