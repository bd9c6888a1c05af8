// Internal header: the FP64 Wilson stencil with the hops of a site spread over lanes, for
// launches with too few (site, RHS) pairs to fill the GPU one thread each.
//
// Same operator, layouts and epilogues as dslash.cu.  There one thread walks the eight hops
// of a site: on a small lattice that is one long serial chain on a few SMs (4^4: two blocks;
// GB300 issues an FP64 warp instruction about every 64 cycles, so the ~900 FP64 instructions
// of a site took 37 us with 150 SMs idle).  Here 16 lanes share a (site, RHS): lane
// 2 h + s forms spin component s of the half spinor of hop h (three colours), multiplies it
// by the link and leaves the product in shared memory; lanes 0..11 then each sum one
// complex component of the output over the eight hops and run the epilogue on it.  The
// arithmetic per site is the same but for the reduction, about 34 FP64 warp instructions
// per site against 28.5, so the one-thread form stays for lattices that fill the GPU.
#pragma once
#include <cstring>

#include "cg_scalars.cuh"
#include "fastdiv.h"
#include "kernels.cuh"

namespace eig {

struct SplitArgs {
    const void *in;
    void *out;
    const void *cen;  // centre-term input (odd-even form), else in; null: hops only
    void *r;
    const void *b;    // residual epilogue
    void *tsave;
    const void *g;
    // complex-component, site and RHS strides of in and out, so that the natural layout
    // of the API can be read and written as it is
    unsigned in_c, in_x, in_r, out_c, out_x, out_r;
    unsigned L0, L1, L2, L3, V, Vg, lh;
    FastDiv d0, d1, d2, dh;
    int eo;
    unsigned k, kshift;
    double diag, hcoef;
    int save_t, set_rho;
    CGScalars *st;
    double *h_alpha, *h_beta, *h_rho;
    int iter;
    const int *jbase;
    double *partials;
    unsigned *counter;
};

// largest number of (site, RHS) pairs the split launchers take (32-bit offsets)
constexpr long SPLIT_MAX = 1L << 20;

namespace {

// complex component e of the spinor at offset o = site stride * site + RHS stride * RHS,
// component stride cs
__device__ __forceinline__ Cx<double> load_comp(const void *p, unsigned cs, unsigned o, int e) {
    const double2 d = static_cast<const double2 *>(p)[(unsigned)e * cs + o];
    return cmk<double>(d.x, d.y);
}
__device__ __forceinline__ void store_comp(void *p, unsigned cs, unsigned o, int e, Cx<double> z) {
    static_cast<double2 *>(p)[(unsigned)e * cs + o] = make_double2(z.re, z.im);
}

// the rows of the link this lane multiplies by: u[a][b] = U[a][b] (bwd = false) or
// conj(U[b][a]) (bwd = true)
__device__ __forceinline__ void load_link_for(const void *g, unsigned Vg, int mu, unsigned s, bool bwd,
                                              Cx<double> (&u)[3][3]) {
    GaugeView gv;
    gv.data = g;
    gv.V = Vg;
    Link<double> U;
    GaugeLoad<GF_F64_18>::load(gv, mu, s, U);
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
            u[a][b].re = bwd ? U.u[b][a].re : U.u[a][b].re;
            u[a][b].im = bwd ? -U.u[b][a].im : U.u[a][b].im;
        }
}

// What lane l = 2 hop + spin of a 16-lane group does in every site: the projection
// h = a_spin + ph (lower partner), partner spin part, factor +-1 or +-i
struct LaneRole {
    int l, mu, sp, part;
    bool bwd, img;
    double sre, sim;
};
template <bool DAG>
__device__ __forceinline__ LaneRole lane_role(int l) {
    constexpr int SF = DAG ? +1 : -1;  // forward projector I + SF g_mu, backward I - SF g_mu
    LaneRole q;
    q.l = l;
    q.mu = l >> 2;
    q.sp = l & 1;
    q.bwd = (l >> 1) & 1;
    q.part = q.mu <= 1 ? 1 - q.sp : q.sp;
    q.img = q.mu == 0 || q.mu == 2;
    const bool neg = ((q.mu == 1 && q.sp == 0) || (q.mu == 2 && q.sp == 1)) != ((q.bwd ? -SF : SF) < 0);
    q.sre = (neg != q.img) ? -1.0 : 1.0;
    q.sim = neg ? -1.0 : 1.0;
    return q;
}

// Component l (lanes 0..11) of diag * centre + hcoef * (hop sum) at output site s, RHS r, from
// the field a.in (a.cen: its centre term).  Collective over the warp; live is uniform
// over a 16-lane group.  prod: the group's [8][2][3] products.
template <bool DAG>
__device__ __forceinline__ Cx<double> split_component(const SplitArgs &a, const LaneRole &q, bool live, unsigned s, unsigned r,
                                                      Cx<double> (*prod)[2][3]) {
    constexpr int SF = DAG ? +1 : -1;
    const unsigned s1 = a.L0, s2 = a.L0 * a.L1, s3 = s2 * a.L2;
    unsigned x, y, z, tt, sl;
    if (a.eo >= 0) {
        const unsigned rest = a.lh > 1 ? fastdiv(s, a.dh) : s, q2 = fastdiv(rest, a.d1);
        tt = fastdiv(q2, a.d2);
        y = rest - q2 * a.L1;
        z = q2 - tt * a.L2;
        x = 2 * (s - rest * a.lh) + ((a.eo + y + z + tt) & 1);
        sl = x + rest * a.L0;
    } else {
        const unsigned q1 = fastdiv(s, a.d0), q2 = fastdiv(q1, a.d1);
        tt = fastdiv(q2, a.d2);
        x = s - q1 * a.L0;
        y = q1 - q2 * a.L1;
        z = q2 - tt * a.L2;
        sl = s;
    }
    const int l = q.l, mu = q.mu;
    const unsigned cm = mu == 0 ? x : (mu == 1 ? y : (mu == 2 ? z : tt));
    const unsigned Lm = mu == 0 ? a.L0 : (mu == 1 ? a.L1 : (mu == 2 ? a.L2 : a.L3));
    const unsigned sm = mu == 0 ? 1u : (mu == 1 ? s1 : (mu == 2 ? s2 : s3));
    const unsigned nl = q.bwd ? (cm == 0 ? sl + (Lm - 1) * sm : sl - sm) : (cm == Lm - 1 ? sl - (Lm - 1) * sm : sl + sm);
    const unsigned nf = a.eo >= 0 ? nl >> 1 : nl;  // field index of the neighbour
    const unsigned oin = nf * a.in_x + r * a.in_r, oc = s * a.in_x + r * a.in_r;
    Cx<double> c0 = cmk<double>(0, 0);
    if (live) {
        Cx<double> h[3], u[3][3], v[3];
#pragma unroll
        for (int c = 0; c < 3; c++) h[c] = load_comp(a.in, a.in_c, oin, q.sp * 3 + c);
#pragma unroll
        for (int c = 0; c < 3; c++) v[c] = load_comp(a.in, a.in_c, oin, 6 + q.part * 3 + c);
        load_link_for(a.g, a.Vg, mu, q.bwd ? nl : sl, q.bwd, u);
        if (l < 12 && a.cen) c0 = load_comp(a.cen, a.in_c, oc, l);  // in flight with the hops
#pragma unroll
        for (int c = 0; c < 3; c++) {
            h[c].re = fma(q.sre, q.img ? v[c].im : v[c].re, h[c].re);
            h[c].im = fma(q.sim, q.img ? v[c].re : v[c].im, h[c].im);
        }
#pragma unroll
        for (int i = 0; i < 3; i++) {
            Cx<double> w = cmul(u[i][0], h[0]);
            w = cfma(u[i][1], h[1], w);
            w = cfma(u[i][2], h[2], w);
            prod[l >> 1][q.sp][i] = w;
        }
    }
    __syncwarp();
    Cx<double> o = cmk<double>(0, 0);
    if (l < 12 && live) {
        const int so = l / 3, c = l - 3 * so, lo = so & 1;
        Cx<double> acc = cmk<double>(0, 0);
#pragma unroll
        for (int hh = 0; hh < 8; hh++) {
            const int m = hh >> 1, sg = (hh & 1) ? -SF : SF;
            // upper spins take the product, lower spins sg B_mu^H of it
            const int from = so < 2 ? lo : (m <= 1 ? 1 - lo : lo);
            const Cx<double> w = prod[hh][from][c];
            const bool im = so >= 2 && (m == 0 || m == 2);
            bool ng = false;
            if (so >= 2) ng = ((m == 0) || (m == 1 && lo == 1) || (m == 2 && lo == 0)) != (sg < 0);
            // factor (-1)^ng, times i where im
            const double fr = (ng != im) ? -1.0 : 1.0, fi = ng ? -1.0 : 1.0;
            acc.re = fma(fr, im ? w.im : w.re, acc.re);
            acc.im = fma(fi, im ? w.re : w.im, acc.im);
        }
        const double d = a.diag, hc = a.hcoef;
        o = cmk<double>(d * c0.re + hc * acc.re, d * c0.im + hc * acc.im);
    }
    __syncwarp();
    return o;
}

// |component|^2 summed over a 16-lane group (the same in its lanes)
__device__ __forceinline__ double group_norm2(bool mine, Cx<double> o) {
    double n = mine ? o.re * o.re + o.im * o.im : 0.0;
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) n += __shfl_xor_sync(0xffffffffu, n, off);
    return n;
}

// Site s, RHS r through the epilogue (see launch_dslash, _norm, _cg and _resid in kernels.cuh);
// returns the group's |result|^2 (0 for SPL_PLAIN).  Collective over the warp, live uniform over
// a 16-lane group.
template <bool DAG, int EPI>
__device__ __forceinline__ double split_site(const SplitArgs &a, const LaneRole &role, bool live, unsigned s, unsigned r,
                                             Cx<double> (*prod)[2][3]) {
    const int l = role.l;
    const unsigned oo = s * a.out_x + r * a.out_r;
    const bool mine = live && l < 12;
    Cx<double> e0 = cmk<double>(0, 0);
    if (EPI == SPL_CG && mine) e0 = load_comp(a.r, a.out_c, oo, l);
    if (EPI == SPL_RESID && mine) e0 = load_comp(a.b, a.out_c, oo, l);
    Cx<double> o = split_component<DAG>(a, role, live, s, r, prod);
    if (EPI == SPL_RESID) o = e0 - o;
    if (EPI == SPL_CG) {
        const CGScalars &st = a.st[r];
        const double al = st.active ? st.alpha : 0.0;
        if (mine && a.save_t) store_comp(a.tsave, a.V, s, l, o);  // single RHS
        o = cmk<double>(e0.re - al * o.re, e0.im - al * o.im);
    }
    if (mine) store_comp(EPI == SPL_CG || EPI == SPL_RESID ? a.r : a.out, a.out_c, oo, l, o);
    return EPI != SPL_PLAIN ? group_norm2(mine, o) : 0.0;
}

template <bool DAG, int EPI>
__global__ void __launch_bounds__(128) k_dslash_split(const SplitArgs a) {
    __shared__ Cx<double> prod[8][8][2][3];  // [group][hop][spin][colour]
    __shared__ double smem[(128 / 32) * MAX_RHS];
    __shared__ double gsum[8];
    if (EPI == SPL_NORM || EPI == SPL_CG) {
        bool any = false;
        for (unsigned q = 0; q < a.k; q++) any = any || a.st[q].active;
        if (!any) return;
    }
    const int t = threadIdx.x, grp = t >> 4, l = t & 15;
    const LaneRole role = lane_role<DAG>(l);
    const unsigned total = a.V << a.kshift, step = gridDim.x * (blockDim.x >> 4);
    double nrm = 0.0;
    const unsigned niter = (total + step - 1) / step;
    for (unsigned it = 0; it < niter; it++) {
        const unsigned g = it * step + blockIdx.x * (blockDim.x >> 4) + grp;
        const bool live = g < total;  // uniform over a group, not over a warp
        const unsigned s = live ? g >> a.kshift : 0u, r = g & (a.k - 1);
        nrm += split_site<DAG, EPI>(a, role, live, s, r, prod[grp]);  // a group's RHS is the same in every pass
    }
    if (EPI == SPL_PLAIN) return;
    const int ngrp = blockDim.x >> 4, k = (int)a.k;
    if (l == 0) gsum[grp] = nrm;
    __syncthreads();
    if (t < k) {
        double v = 0.0;
        for (int q = 0; q < ngrp; q++)
            if (((blockIdx.x * ngrp + q) & (k - 1)) == t) v += gsum[q];
        a.partials[(long)blockIdx.x * k + t] = v;
    }
    CGScalars *const sts = a.st;
    double *const h_alpha = a.h_alpha, *const h_beta = a.h_beta, *const h_rho = a.h_rho;
    const int iter = a.iter + (a.jbase ? *a.jbase : 0), set_rho = a.set_rho;
    grid_finish_rhs(k, a.partials, a.counter, smem, [=](int rr, double tot) {
        finish_scalars<EPI>(sts, h_alpha, h_beta, h_rho, iter, k, set_rho, rr, tot);
    });
}

inline void split_args(SplitArgs &a, const DslashCall &c) {
    memset(&a, 0, sizeof(a));
    a.in = c.in.v.data;
    a.out = c.out.v.data;
    a.g = c.gauge.data;
    a.L0 = c.L[0];
    a.L1 = c.L[1];
    a.L2 = c.L[2];
    a.L3 = c.L[3];
    a.d0 = fastdiv_make(a.L0);
    a.d1 = fastdiv_make(a.L1);
    a.d2 = fastdiv_make(a.L2);
    a.lh = a.L0 / 2;
    if (a.lh >= 2) a.dh = fastdiv_make(a.lh);
    a.Vg = (unsigned)c.V;
    a.eo = c.eo_parity;
    a.V = (unsigned)(c.eo_parity >= 0 ? c.V / 2 : c.V);
    a.k = (unsigned)c.k;
    while ((1u << a.kshift) < a.k) a.kshift++;
    a.in_c = a.out_c = a.V * a.k;
    a.in_x = a.out_x = a.k;
    a.in_r = a.out_r = 1;
    if (c.nat_in) {  // [rhs][site][component]
        a.in_c = 1;
        a.in_x = 12;
        a.in_r = 12 * a.V;
    }
    if (c.nat_out) {
        a.out_c = 1;
        a.out_x = 12;
        a.out_r = 12 * a.V;
    }
    a.cen = c.in.v.data;
    if (c.eo_parity >= 0) a.cen = c.cen.v.data;
    a.diag = c.diag;
    a.hcoef = c.hcoef;
}

inline void split_reduction(SplitArgs &a, CGScalars *st, const History &h, int iter, const RedScratch &red) {
    a.st = st;
    a.h_alpha = h.alpha;
    a.h_beta = h.beta;
    a.h_rho = h.rho;
    a.iter = iter;
    a.jbase = h.jbase;
    a.partials = red.partials;
    a.counter = red.counter;
}

// Blocks of one warp while there are fewer warps than SMs (each then has an SM's FP64 units
// to itself), of four otherwise; 16 resident warps per SM at most, and a multiple of 16
// blocks when a block makes several passes, so that a group keeps its RHS from pass to pass.
template <int EPI>
cudaError_t split_launch(bool dag, const SplitArgs &a, int cap, cudaStream_t s) {
    const long groups = (long)a.V << a.kshift, warps = (groups + 1) / 2;
    if (groups > SPLIT_MAX || a.k > (unsigned)MAX_RHS) return cudaErrorInvalidValue;
    const int sms = device_sm_count();
    const int tpb = warps <= sms ? 32 : (warps <= 2L * sms ? 64 : 128);
    const long need = (groups + tpb / 16 - 1) / (tpb / 16);
    long most = (long)sms * (2048 / tpb) / 4;
    if (cap > 0 && most > cap) most = cap;
    long grid = need;
    if (grid > most) grid = most / 16 * 16;
    if (grid < 1) grid = need < 16 ? need : 16;
    if (dag) k_dslash_split<true, EPI><<<(int)grid, tpb, 0, s>>>(a);
    else k_dslash_split<false, EPI><<<(int)grid, tpb, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace
}  // namespace eig
