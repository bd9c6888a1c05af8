// CG iterations on small FP32 lattices inside one thread-block cluster.
//
// On a lattice of a few thousand sites a CG iteration of three launches (p update, u = M p,
// t = M^H u) is a chain of latencies: the launches, eight dependent rounds of L2 loads per
// stencil in a few warps, and a last block that sums each reduction (8^4, one RHS: 18 us per
// iteration replayed from a graph, 6 us per kernel).  Spreading the sites over more SMs does not
// help: a grid-wide barrier through L2 cost more than the launch it replaced (21 us per
// iteration with three of them in one cooperative launch).  Here 16 SMs hold the whole problem:
// one cluster of 16 CTAs, one thread per (site, RHS), p, u and the links in shared memory, r and
// x in registers, neighbours read through distributed shared memory, and the cluster barrier
// (hardware) orders the phases.  Reductions go the same way: warps or CTAs store their sums into
// every CTA's shared memory, and all add them up in the same order, so alpha, beta and the
// stopping decisions are the same everywhere.  One launch runs up to 16 iterations; CTA 0 keeps
// the device scalars.
//
// 8^4, one RHS: 13.6 us per iteration (whole solve to 1e-8 at cond 1e4: 5.2 -> 4.0 ms); 4^4: 9.1.
// Of about ten cycles per issue of a warp 3.1 wait for loads through distributed shared memory, 2.8
// for the barriers and their release, at two warps per sub-partition; the FP64 sums and divisions of
// the two reductions keep their pipes active for 1.2 us (profiles/cg_cluster_8x8.md).  Nothing in
// the loop touches global memory but the window: the barrier's release waits for global stores, and its acquire drops the links
// from L1 (with the links and x in global memory an iteration took 15.5 us).  Beyond 4096 (site,
// RHS) pairs a thread would hold two and the graph of three launches is as fast (8^4, k = 2: 25
// us per iteration).  Up to there the cluster is the faster one at every width (us per iteration,
// cluster : graph): 4^4, k = 1 10.1 : 17.4, k = 4 11.6 : 20.1, k = 8 14.8 : 22.1, k = 16 22.1 : 26.3;
// 4^3x8, k = 8 17.0 : 21.9; 4x8^3, k = 2 14.6 : 20.1; 8^4, k = 1 14.4 : 18.1 (EIG_CG_CLUSTER=0).
//
// Steps, scalars and their order are those of launch_pupdate, launch_dslash_norm and
// launch_dslash_cg (kernels.cuh), the arithmetic that of dslash32.cuh.
#include <algorithm>
#include <cstring>

#include "cg_scalars.cuh"
#include "device_cache.h"
#include "dslash32.cuh"
#include "prof.h"

namespace eig {

namespace {

constexpr int CL = 16;       // CTAs of the cluster
constexpr int CL_T = 256;    // threads per CTA at most (255 registers each)
static_assert(CG_CLUSTER_MAX == (long)CL * CL_T, "one (site, RHS) per thread");

struct ClusterArgs {
    const void *g;
    float4 *p, *r, *x;
    unsigned L0, L1, L2, L3, V, n, k, kshift;
    FastDiv d0, d1, d2;
    float diag, hcoef;
    CGScalars *st;
    double *h_alpha, *h_beta, *h_rho;
    int j0, iters, first;
    // eigCG window (one RHS): iteration j0 + 1 + q appends to win + slot[q]; the last
    // iteration's t goes to tsave if given
    char *win;
    size_t slot_bytes;
    int slot[CG_CLUSTER_ITERS];
    float4 *tsave;
};

__device__ __forceinline__ uint32_t cl_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cl_map(uint32_t smem_addr, uint32_t cta) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(cta));
    return r;
}
// volatile: ordered with the barriers, but free to run ahead of arithmetic
__device__ __forceinline__ float4 cl_ld(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(addr));
    return v;
}
__device__ __forceinline__ float2 cl_ld2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ void cl_st(uint32_t addr, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
// every thread of the cluster; orders shared-memory accesses before it with those after it
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void cl_load(uint32_t addr, uint32_t plane, float4 (&v)[6]) {
#pragma unroll
    for (int c = 0; c < 6; c++) v[c] = cl_ld(addr + c * plane);
}
__device__ __forceinline__ void cl_unpack(const float4 (&d)[6], Sp &v) {
#pragma unroll
    for (int c = 0; c < 6; c++) {
        v.c[2 * c] = f2(d[c].x, d[c].y);
        v.c[2 * c + 1] = f2(d[c].z, d[c].w);
    }
}

// links in shared memory, planes over the CTA's sites: per direction 3 planes of float4 (12
// reals) or 9 of float2 (18 reals), as in global memory
template <int GF>
struct ClLink;
template <>
struct ClLink<GF_F32_12> {
    static constexpr int PLANES = 3, BYTES = 16;
    float4 v[3];
    __device__ __forceinline__ void load(uint32_t addr, uint32_t plane) {
#pragma unroll
        for (int c = 0; c < 3; c++) v[c] = cl_ld(addr + c * plane);
    }
    __device__ __forceinline__ void unpack(Lk &U) const {
        U.u[0] = f2(v[0].x, v[0].y);
        U.u[1] = f2(v[0].z, v[0].w);
        U.u[2] = f2(v[1].x, v[1].y);
        U.u[3] = f2(v[1].z, v[1].w);
        U.u[4] = f2(v[2].x, v[2].y);
        U.u[5] = f2(v[2].z, v[2].w);
        rebuild_row2(U);
    }
};
template <>
struct ClLink<GF_F32_18> {
    static constexpr int PLANES = 9, BYTES = 8;
    float2 v[9];
    __device__ __forceinline__ void load(uint32_t addr, uint32_t plane) {
#pragma unroll
        for (int c = 0; c < 9; c++) v[c] = cl_ld2(addr + c * plane);
    }
    __device__ __forceinline__ void unpack(Lk &U) const {
#pragma unroll
        for (int e = 0; e < 9; e++) U.u[e] = v[e];
    }
};

// where a thread finds its eight neighbours (chunk 0 of p), its own chunk 0, and the links of
// its hops (plane 0 of direction mu): shared::cluster addresses
struct ClAddr {
    uint32_t nbr[8], cen, lk[8];
    uint32_t plane, lplane;  // bytes between planes of a field, of the links
};

template <int MU, int SG, bool DAGGER, int GF>
__device__ __forceinline__ void cl_hop(const float4 (&d)[6], const ClLink<GF> &l, Sp &acc) {
    Lk U;
    Sp nb;
    Hf h, uh;
    l.unpack(U);
    cl_unpack(d, nb);
    project<MU, SG>(nb, h);
    mul_link<DAGGER>(U, h, uh);
    accumulate<MU, SG>(acc, uh);
}

// out = diag * centre + hcoef * (hop sum) of the field `off` bytes behind p; hop h + 1 loads
// while hop h is computed
template <bool DAG, int GF>
__device__ __forceinline__ void cl_stencil(const ClusterArgs &a, const ClAddr &ad, uint32_t off, Sp &out) {
    constexpr int SF = DAG ? +1 : -1, SB = -SF;
    Sp acc;
#pragma unroll
    for (int e = 0; e < 12; e++) acc.c[e] = f2(0.f, 0.f);
    float4 d[2][6];
    ClLink<GF> l[2];
    cl_load(ad.nbr[0] + off, ad.plane, d[0]);
    l[0].load(ad.lk[0], ad.lplane);
#pragma unroll
    for (int h = 0; h < 8; h++) {
        const int cur = h & 1, nx = cur ^ 1;
        if (h < 7) {
            cl_load(ad.nbr[h + 1] + off, ad.plane, d[nx]);
            l[nx].load(ad.lk[h + 1], ad.lplane);
        } else {
            cl_load(ad.cen + off, ad.plane, d[nx]);
        }
        switch (h) {
            case 0: cl_hop<0, SF, false>(d[cur], l[cur], acc); break;
            case 1: cl_hop<0, SB, true>(d[cur], l[cur], acc); break;
            case 2: cl_hop<1, SF, false>(d[cur], l[cur], acc); break;
            case 3: cl_hop<1, SB, true>(d[cur], l[cur], acc); break;
            case 4: cl_hop<2, SF, false>(d[cur], l[cur], acc); break;
            case 5: cl_hop<2, SB, true>(d[cur], l[cur], acc); break;
            case 6: cl_hop<3, SF, false>(d[cur], l[cur], acc); break;
            default: cl_hop<3, SB, true>(d[cur], l[cur], acc); break;
        }
    }
    Sp c0;
    cl_unpack(d[0], c0);
    const F2 d2 = f2(a.diag, a.diag), mh = f2(a.hcoef, a.hcoef);
#pragma unroll
    for (int e = 0; e < 12; e++) out.c[e] = fma2(mh, acc.c[e], mul2(d2, c0.c[e]));
}

__device__ __forceinline__ float4 chunk_of(const Sp &v, int c) {
    return make_float4(v.c[2 * c].x, v.c[2 * c].y, v.c[2 * c + 1].x, v.c[2 * c + 1].y);
}

template <int GF>
__global__ void __launch_bounds__(CL_T, 1) k_cg_cluster(const ClusterArgs a) {
    extern __shared__ __align__(16) float4 fld[];  // p: 6 planes of T, then u, then the links
    __shared__ double slots[2][CL * MAX_RHS], wsum[(CL_T / 32) * MAX_RHS];
    static_assert(MAX_RHS >= 8, "slots hold 8 warps' sums of one RHS");
    __shared__ CGScalars sc[MAX_RHS];
    __shared__ float s_inv;
    const unsigned T = blockDim.x, t = threadIdx.x, cta = cl_rank();
    const int lane = t & 31, warp = t >> 5, k = (int)a.k, nw = (int)(T >> 5);
    const unsigned g = cta * T + t, TS = T >> a.kshift;  // sites per CTA (T is a multiple of k)
    const bool live = g < a.n;
    const unsigned ge = live ? g : 0u, s = ge >> a.kshift, r = ge & (a.k - 1);
    const int q = t & (k - 1);  // this thread's RHS, live or not
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(fld), lbase = base + 12 * T * 16;
    using LK = ClLink<GF>;
    ClAddr ad;
    ad.plane = T * 16;
    ad.lplane = TS * LK::BYTES;
    {
        const unsigned q1 = fastdiv(s, a.d0), q2 = fastdiv(q1, a.d1), tt = fastdiv(q2, a.d2);
        const unsigned c[4] = {s - q1 * a.L0, q1 - q2 * a.L1, q2 - tt * a.L2, tt};
        const unsigned L[4] = {a.L0, a.L1, a.L2, a.L3}, st[4] = {1u, a.L0, a.L0 * a.L1, a.L0 * a.L1 * a.L2};
#pragma unroll
        for (int mu = 0; mu < 4; mu++) {
            const unsigned f = c[mu] == L[mu] - 1 ? s - (L[mu] - 1) * st[mu] : s + st[mu];
            const unsigned b = c[mu] == 0 ? s + (L[mu] - 1) * st[mu] : s - st[mu];
            const unsigned ef = (f << a.kshift) + r, eb = (b << a.kshift) + r;
            const uint32_t lm = lbase + mu * LK::PLANES * ad.lplane;
            ad.nbr[2 * mu] = cl_map(base + (ef % T) * 16, ef / T);
            ad.nbr[2 * mu + 1] = cl_map(base + (eb % T) * 16, eb / T);
            ad.lk[2 * mu] = cl_map(lm + (s % TS) * LK::BYTES, s / TS);
            ad.lk[2 * mu + 1] = cl_map(lm + (b % TS) * LK::BYTES, b / TS);
        }
        ad.cen = cl_map(base + t * 16, cta);
    }
    float4 rr[6], xx[6];
#pragma unroll
    for (int c = 0; c < 6; c++) {
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
        rr[c] = xx[c] = d;
        if (live) {
            d = a.p[(size_t)c * a.n + g];
            rr[c] = a.r[(size_t)c * a.n + g];
            xx[c] = a.x[(size_t)c * a.n + g];
        }
        fld[c * T + t] = d;
        fld[(6 + c) * T + t] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    {  // the links of the CTA's sites
        unsigned char *lf = reinterpret_cast<unsigned char *>(fld + 12 * T);
        for (unsigned i = t; i < 4 * LK::PLANES * TS; i += T) {
            const unsigned pl = i / TS, ls = cta * TS + (i - pl * TS);
            if (ls >= a.V) continue;
            if (LK::BYTES == 16)
                reinterpret_cast<float4 *>(lf)[i] = __ldg(static_cast<const float4 *>(a.g) + (size_t)pl * a.V + ls);
            else
                reinterpret_cast<float2 *>(lf)[i] = __ldg(static_cast<const float2 *>(a.g) + (size_t)pl * a.V + ls);
        }
    }
    if ((int)t < k) sc[t] = a.st[t];
    cl_sync();
    auto any_active = [&]() {
        bool any = false;
        for (int i = 0; i < k; i++) any = any || sc[i].active;
        return any;
    };
    // the cluster's sum of v per RHS, in lanes < k of warp 0.  Few sums: every warp stores its own
    // into every CTA (an FP64 shuffle tree before the barrier and one after; an FP64 add costs
    // ~100 cycles here); many: the CTA's warps are added up first (4^4, k = 16: 21.7 against 25.8
    // us per iteration; 8^4, k = 1: 14.4 against 13.6).  The barrier inside also publishes the
    // shared-memory fields.
    const bool by_warp = nw * k <= 8;
    const int per_cta = by_warp ? nw : 1;  // sums of one RHS that a CTA contributes
    auto cl_sum = [&](float site, int which) {
        double v = live ? (double)site : 0.0;
        for (int off = 16; off >= k; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (!by_warp) {
            if (lane < k) wsum[warp * k + lane] = v;
            __syncthreads();
            if (warp == 0) {
                v = 0.0;
                for (int i = lane; i < nw * k; i += 32) v += wsum[i];
                for (int off = 16; off >= k; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            }
        }
        if (by_warp || warp == 0) {
            const uint32_t mine =
                (uint32_t)__cvta_generic_to_shared(&slots[which][(cta * per_cta + (by_warp ? warp : 0)) * k + (lane & (k - 1))]);
            for (int i = lane; i < CL * k; i += 32) cl_st(cl_map(mine, i >> a.kshift), v);
        }
        cl_sync();
        v = 0.0;
        if (warp == 0) {
            for (int i = lane; i < CL * per_cta * k; i += 32) v += slots[which][i];
            for (int off = 16; off >= k; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        }
        return v;
    };
    for (int it = 0; it < a.iters; it++) {
        if (!any_active()) break;  // the same in every CTA
        const int j = a.j0 + 1 + it;
        const bool first = a.first && it == 0;
        if (a.win) {
            if (t == 0) s_inv = (float)(1.0 / sqrt(sc[0].rho));
            __syncthreads();
        }
        // p update: x += alpha p of the previous iteration, p = r + beta p, window append
        const bool active = sc[q].active, pend = !first && sc[q].x_pending;
        if (live && (first || active || pend)) {
            const float al = (float)sc[q].alpha, be = (float)sc[q].beta;
#pragma unroll
            for (int c = 0; c < 6; c++) {
                float4 pp = fld[c * T + t];
                const float4 rc = rr[c];
                if (pend) {
                    xx[c].x += al * pp.x;
                    xx[c].y += al * pp.y;
                    xx[c].z += al * pp.z;
                    xx[c].w += al * pp.w;
                }
                if (first) pp = rc;
                else if (active) pp = make_float4(rc.x + be * pp.x, rc.y + be * pp.y, rc.z + be * pp.z, rc.w + be * pp.w);
                if (first || active) fld[c * T + t] = pp;
                if (a.win && active) {
                    const float inv = s_inv;
                    reinterpret_cast<float4 *>(a.win + (size_t)a.slot[it] * a.slot_bytes)[(size_t)c * a.n + g] =
                        make_float4(rc.x * inv, rc.y * inv, rc.z * inv, rc.w * inv);
                }
            }
        }
        cl_sync();
        // u = M p, alpha = rho / ||u||^2
        {
            Sp u;
            cl_stencil<false, GF>(a, ad, 0u, u);
#pragma unroll
            for (int c = 0; c < 6; c++) fld[(6 + c) * T + t] = chunk_of(u, c);
            const double tot = cl_sum(norm2f(u), 0);
            if ((int)t < k) finish_scalars<SPL_NORM>(sc, a.h_alpha, a.h_beta, a.h_rho, j, k, 0, t, tot);
            __syncthreads();
        }
        if (!any_active()) break;
        // t = M^H u, r -= alpha t, rho and beta
        {
            Sp tv;
            cl_stencil<true, GF>(a, ad, 6 * ad.plane, tv);
            const float al = sc[q].active ? (float)sc[q].alpha : 0.f;
            const F2 mal = f2(-al, -al);
            if (a.tsave && it == a.iters - 1 && live)
#pragma unroll
                for (int c = 0; c < 6; c++) a.tsave[(size_t)c * a.n + g] = chunk_of(tv, c);
            Sp rn;
#pragma unroll
            for (int c = 0; c < 6; c++) {
                rn.c[2 * c] = fma2(mal, tv.c[2 * c], f2(rr[c].x, rr[c].y));
                rn.c[2 * c + 1] = fma2(mal, tv.c[2 * c + 1], f2(rr[c].z, rr[c].w));
                rr[c] = chunk_of(rn, c);
            }
            const double tot = cl_sum(norm2f(rn), 1);
            if ((int)t < k) finish_scalars<SPL_CG>(sc, a.h_alpha, a.h_beta, a.h_rho, j, k, 0, t, tot);
            __syncthreads();
        }
    }
    if (live)
#pragma unroll
        for (int c = 0; c < 6; c++) {
            a.p[(size_t)c * a.n + g] = fld[c * T + t];
            a.r[(size_t)c * a.n + g] = rr[c];
            a.x[(size_t)c * a.n + g] = xx[c];
        }
    if (cta == 0 && (int)t < k) a.st[t] = sc[t];
    cl_sync();  // no CTA leaves while another may still read its shared memory
}

using ClusterKernel = void (*)(ClusterArgs);

ClusterKernel cluster_kernel(int gformat) {
    return gformat == GF_F32_12 ? k_cg_cluster<GF_F32_12> : (gformat == GF_F32_18 ? k_cg_cluster<GF_F32_18> : nullptr);
}

// launch configuration of n (site, RHS) pairs, k RHS; attr must outlive cfg
void cluster_config(long n, int k, int gformat, cudaStream_t s, cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr) {
    const unsigned T = (unsigned)(((n + CL - 1) / CL + 31) / 32 * 32);
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(CL);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = (size_t)12 * T * sizeof(float4) + (size_t)(gformat == GF_F32_12 ? 192 : 288) * (T / k);
    cfg.stream = s;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = CL;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
}

// a cluster of 16 and its shared memory are opt-ins, per device; those of the largest CTAs, so that one
// setting does for every launch
cudaError_t cluster_attributes(int gformat) {
    const void *kern = (const void *)cluster_kernel(gformat);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    cluster_config(CG_CLUSTER_MAX, 1, gformat, 0, cfg, attr);
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes);
}

// whether the current GPU can hold a cluster of 16 with the largest CTAs (asked, and the opt-ins set,
// once per device)
bool cluster_fits(int gformat) {
    static DeviceCache fits[2];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    return fits[gformat == GF_F32_12 ? 0 : 1].get(dev, [&] {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        cluster_config(CG_CLUSTER_MAX, 1, gformat, 0, cfg, attr);
        int clusters = 0;
        cudaError_t e = cluster_attributes(gformat);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveClusters(&clusters, (const void *)cluster_kernel(gformat), &cfg);
        cudaGetLastError();
        return e == cudaSuccess ? (clusters >= 1 ? 1 : 0) : -1;
    });
}

}  // namespace

bool cg_cluster_takes(const DslashCall &c) {
    return c.eo_parity < 0 && c.in.prec == P32 && c.V * c.k <= CG_CLUSTER_MAX && cluster_kernel(c.gformat) &&
           cluster_fits(c.gformat);
}

cudaError_t launch_cg_cluster(const DslashCall &c, const CgCluster &q, CGScalars *st, History h, cudaStream_t s) {
    if (!cg_cluster_takes(c) || q.n < 1 || q.n > CG_CLUSTER_ITERS || (q.win && c.k != 1)) return cudaErrorInvalidValue;
    // p, r and x in and out and the links once; the window append per iteration
    ProfScope prof("cg_cluster", (double)c.V * (c.gformat == GF_F32_12 ? 192 : 288) + (double)c.V * c.k * 6 * 96 +
                                     (q.win ? (double)q.n * c.V * 96 : 0.0), s);
    ClusterArgs a;
    memset(&a, 0, sizeof(a));
    a.g = c.gauge.data;
    a.p = static_cast<float4 *>(q.p.v.data);
    a.r = static_cast<float4 *>(q.r.v.data);
    a.x = static_cast<float4 *>(q.x.v.data);
    a.L0 = c.L[0];
    a.L1 = c.L[1];
    a.L2 = c.L[2];
    a.L3 = c.L[3];
    a.d0 = fastdiv_make(a.L0);
    a.d1 = fastdiv_make(a.L1);
    a.d2 = fastdiv_make(a.L2);
    a.V = (unsigned)c.V;
    a.k = (unsigned)c.k;
    while ((1u << a.kshift) < a.k) a.kshift++;
    a.n = a.V << a.kshift;
    a.diag = (float)c.diag;
    a.hcoef = (float)c.hcoef;
    a.st = st;
    a.h_alpha = h.alpha;
    a.h_beta = h.beta;
    a.h_rho = h.rho;
    a.j0 = q.j0;
    a.iters = q.n;
    a.first = q.first;
    a.win = static_cast<char *>(q.win);
    a.slot_bytes = q.slot_bytes;
    for (int i = 0; i < q.n; i++) a.slot[i] = q.slot[i];
    a.tsave = static_cast<float4 *>(q.tsave);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    cluster_config((long)a.n, c.k, c.gformat, s, cfg, attr);
    return cudaLaunchKernelEx(&cfg, cluster_kernel(c.gformat), a);
}

}  // namespace eig
