// The FP64 Wilson stencil in block fixed-point integer arithmetic.
//
// GB300 issues an FP64 warp instruction about every 64 cycles per SM sub-partition, so the
// ~912 FP64 instructions of a site keep the FP64 units busy for ~1800 cycles per (site, RHS)
// while everything else idles (24^3x64, k = 16: 22.7 ms per product, 4% of HBM).  The integer
// pipes run 32 times faster.  Here the hops are computed on 64-bit integers with one exponent
// per site and RHS (fxmath.h):
//   k_to_fx      brings a field to integers I = x 2^(1079 - e), |I| <= 2^57, e the largest
//                exponent of the 24 reals of a (site, RHS); FP64 bits beyond the 57 below a
//                site's largest component are dropped;
//   k_dslash_fx  projects the eight neighbours of a site by integer adds, aligns the half spinors
//                to their largest exponent (a shift), multiplies by the links (two 29-bit limbs per
//                real, three wide multiply-adds per real product), sums the eight hops exactly
//                and rounds once to FP64, where the centre term and the epilogue are formed.
// The errors are at most 2^-50 of the largest neighbour component, so an element whose hop
// products are all small against that one is not kept (fxmath.h has the bound and the guard): the
// warp forms it again in FP64, 16 lanes to an element (dslash_split.cuh).  The same path takes
// elements with an Inf or NaN among their neighbours, and those near the ends of the exponent
// range.  Links are held relative to a power of two for which the sums of eight hops stay below
// 2^63 (link_scale, found when an operator is created).  Operators whose links differ too much in
// size keep the FP64 stencil, and so do launches too small to fill the GPU (FX_MIN).
//
// What bounds it now: the wide multiply-adds (1728 per site, 2 cycles each on the heavy half of
// the FMA pipe), integer ALU and the latency of the neighbour loads at 16 warps per SM.  Measured
// per product, conversion included (the conversion alone 28 us, 5.4 TB/s):
//   16^3x32, k = 4    FP64 850 us    fixed point 255 us (every element left to FP64: 1135 us)
//   24^3x64, k = 16   FP64 22.8 ms   fixed point 6.34 ms; with the norm, CG and residual epilogues 7.4,
//                     8.5 and 8.0 ms
//   12^3x24, k = 8    double-float (44 bits; used for residual replacements before) 194 us plus
//                     120 us of field conversions per A; fixed point 171 us
// The guard keeps one bit per product (sums of magnitudes in six registers: 303 us at 16^3x32).  Aligning
// the 24 components of a neighbour instead of the 12 of its half spinor, separate sums of the middle
// limbs and conjugating the links one by one took 282 us, and 8.6 ms for the residual at 24^3x64.
// Four blocks per SM (128 registers, 32 to 76 bytes spilled) beat three and two (294 and 377 us when
// four took 282); without the L1 prefetch of the next hop three took 311 us; with the eight hops
// unrolled, 685.
#include <cmath>
#include <cstring>

#include "dslash_split.cuh"
#include "fxmath.h"
#include "kernels.cuh"
#include "prof.h"

namespace eig {

namespace {

// Layout of the integer field and links: tiles of 32 elements ((site, RHS) pairs; sites),
// [element / 32][component][element % 32], so that a warp's loads are contiguous and the
// components of an element sit at fixed distances from one address.
constexpr int TILE = 32;
__host__ __device__ constexpr size_t tiled(unsigned i, int comps) {
    return (size_t)(i / TILE) * (size_t)(TILE * comps) + i % TILE;
}

struct FxArgs {
    const longlong2 *fx;  // hop input in fixed point (re, im), tiled, 12 components
    const int *ex;        // its exponent words: [V][k]
    const int4 *g;        // links, limbs (re hi, re lo, im hi, im lo): [mu] tiled, 9 components
    int gscale;           // ... of links 2^-gscale
    SplitArgs s;          // the call in FP64
};

constexpr int FX_TPB = 128;

__global__ void __launch_bounds__(FX_TPB) k_to_fx(const double2 *__restrict__ in, longlong2 *__restrict__ fxo,
                                                  int *__restrict__ ex, unsigned n) {
    for (unsigned o = blockIdx.x * FX_TPB + threadIdx.x; o < n; o += gridDim.x * FX_TPB) {
        double2 v[12];
#pragma unroll
        for (int c = 0; c < 12; c++) v[c] = in[(size_t)c * n + o];
        unsigned top = 0;  // largest high word, sign removed: its exponent field is the block's
#pragma unroll
        for (int c = 0; c < 12; c++) {
            top = max(top, (unsigned)__double2hiint(v[c].x) & 0x7fffffffu);
            top = max(top, (unsigned)__double2hiint(v[c].y) & 0x7fffffffu);
        }
        const int e = max((int)(top >> 20), 1);
        unsigned spins = 0;
#pragma unroll
        for (int sp = 0; sp < 4; sp++) {
            unsigned any = 0;
#pragma unroll
            for (int c = 3 * sp; c < 3 * sp + 3; c++)
                any |= (unsigned)(__double2loint(v[c].x) | __double2loint(v[c].y)) |
                       (((unsigned)__double2hiint(v[c].x) | (unsigned)__double2hiint(v[c].y)) & 0x7fffffffu);
            spins |= any ? 1u << sp : 0u;
        }
        ex[o] = e | (int)(spins << fx::NZ);
        if (e >= fx::SPECIAL) continue;  // never read
#pragma unroll
        for (int c = 0; c < 12; c++) {
            longlong2 z;
            z.x = fx::to_fixed(v[c].x, e);
            z.y = fx::to_fixed(v[c].y, e);
            fxo[tiled(o, 12) + c * TILE] = z;
        }
    }
}

__host__ __device__ constexpr size_t fx_link_plane(unsigned V) { return (size_t)((V + TILE - 1) / TILE) * TILE * 9; }

// high words of the largest and of the smallest nonzero squared norm of a row or column of the links
// [mu][9][V] (Inf and NaN are above all others); range[0] starts as 0, range[1] as the largest word
__global__ void k_links_range(const double2 *__restrict__ g, unsigned V, unsigned *range) {
    unsigned top = 0, bottom = 0xffffffffu;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < 4u * V; i += gridDim.x * blockDim.x) {
        const unsigned mu = i / V, s = i - mu * V;
        const double2 *p = g + (size_t)mu * 9 * V + s;
        double norm[6] = {0, 0, 0, 0, 0, 0};
        for (int e = 0; e < 9; e++) {
            const double2 u = p[(size_t)e * V];
            const double n = u.x * u.x + u.y * u.y;
            norm[e / 3] += n;
            norm[3 + e % 3] += n;
        }
        for (int q = 0; q < 6; q++) {
            const unsigned w = (unsigned)__double2hiint(norm[q]) & 0x7fffffffu;
            top = max(top, w);
            if (w) bottom = min(bottom, w);
        }
    }
    top = __reduce_max_sync(0xffffffffu, top);
    bottom = __reduce_min_sync(0xffffffffu, bottom);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(range, top);
        atomicMin(range + 1, bottom);
    }
}

// links [mu][9][V] FP64 -> limbs of u 2^(58 - scale)
__global__ void k_links_fx(const double2 *__restrict__ g, int4 *__restrict__ out, unsigned V, double unit) {
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < 4u * V; i += gridDim.x * blockDim.x) {
        const unsigned mu = i / V, s = i - mu * V;
        const double2 *p = g + (size_t)mu * 9 * V + s;
        for (int e = 0; e < 9; e++) {
            const double2 u = p[(size_t)e * V];
            int4 l;
            fx::limbs(__double2ll_rn(u.x * unit), l.x, l.y);
            fx::limbs(__double2ll_rn(u.y * unit), l.z, l.w);
            out[mu * fx_link_plane(V) + tiled(s, 9) + e * TILE] = l;
        }
    }
}

struct I2 {
    long long re, im;
};

__device__ __forceinline__ I2 add(I2 x, I2 y) {
    x.re += y.re;
    x.im += y.im;
    return x;
}
__device__ __forceinline__ I2 sub(I2 x, I2 y) {
    x.re -= y.re;
    x.im -= y.im;
    return x;
}
__device__ __forceinline__ I2 addi(I2 x, I2 y) {  // x + i y
    x.re -= y.im;
    x.im += y.re;
    return x;
}
__device__ __forceinline__ I2 subi(I2 x, I2 y) {  // x - i y
    x.re += y.im;
    x.im -= y.re;
    return x;
}

__device__ __forceinline__ void prefetch_hop_fx(const FxArgs &a, int mu, unsigned o, unsigned ls) {
    const longlong2 *f = a.fx + tiled(o, 12);
#pragma unroll
    for (int e = 0; e < 12; e++) asm volatile("prefetch.global.L1 [%0];" ::"l"(f + e * TILE));
    const int4 *g = a.g + mu * fx_link_plane(a.s.Vg) + tiled(ls, 9);
#pragma unroll
    for (int e = 0; e < 9; e++) asm volatile("prefetch.global.L1 [%0];" ::"l"(g + e * TILE));
}

// One hop: neighbour at field index o (in (site, RHS) units), link (mu, ls),
// conj(U)^T if bwd, projector I + sg g_mu.  mu, bwd and sg are uniform over the launch's
// threads and not template arguments: only the projection and the rebuilding differ between the
// eight hops, and with all of them unrolled the ~11 000 instructions of a site did not fit the
// instruction caches (stalled on instruction fetch 3.8 of 7 cycles per issue).  large: bit e
// is set if product e passes guard_large.
__device__ __forceinline__ void hop_fx(const FxArgs &a, int mu, bool bwd, bool plus, unsigned o, unsigned ls, int sh,
                                       I2 (&acc)[12], unsigned &large) {
    const longlong2 *f = a.fx + tiled(o, 12);
    I2 v[12];
#pragma unroll
    for (int e = 0; e < 12; e++) {
        const longlong2 d = __ldg(f + e * TILE);
        v[e].re = d.x;
        v[e].im = d.y;
    }
    // project: h = a + sg B_mu b (see dslash.cu for B_mu)
    I2 h[6];
    const int which = mu * 2 + (plus ? 1 : 0);
#define FX_PROJECT(F0, B0, F1, B1)                   \
    do {                                             \
        h[0] = F0(v[0], v[B0]);                      \
        h[1] = F0(v[1], v[B0 + 1]);                  \
        h[2] = F0(v[2], v[B0 + 2]);                  \
        h[3] = F1(v[3], v[B1]);                      \
        h[4] = F1(v[4], v[B1 + 1]);                  \
        h[5] = F1(v[5], v[B1 + 2]);                  \
    } while (0)
    switch (which) {
        case 0: FX_PROJECT(subi, 9, subi, 6); break;
        case 1: FX_PROJECT(addi, 9, addi, 6); break;
        case 2: FX_PROJECT(add, 9, sub, 6); break;
        case 3: FX_PROJECT(sub, 9, add, 6); break;
        case 4: FX_PROJECT(subi, 6, addi, 9); break;
        case 5: FX_PROJECT(addi, 6, subi, 9); break;
        case 6: FX_PROJECT(sub, 6, sub, 9); break;
        default: FX_PROJECT(add, 6, add, 9); break;
    }
#undef FX_PROJECT
    int rh[6], rl[6], ih[6], il[6];
#pragma unroll
    for (int e = 0; e < 6; e++) {
        fx::limbs(fx::align(h[e].re, sh), rh[e], rl[e]);
        fx::limbs(fx::align(h[e].im, sh), ih[e], il[e]);
    }
    const int sgn = bwd ? 1 : -1;  // of the links' imaginary parts in the real sums (bwd: conjugate links)
    const int4 *g = a.g + mu * fx_link_plane(a.s.Vg) + tiled(ls, 9);
    const int sq = bwd ? TILE : 3 * TILE, sb = bwd ? 3 * TILE : TILE;
    I2 w[6];
#pragma unroll
    for (int q = 0; q < 3; q++) {
        // output colour q of both spins: sum over colours b of U[q][b] h_b, or conj(U[b][q]) h_b
        int4 u[3];
#pragma unroll
        for (int b = 0; b < 3; b++) {
            u[b] = __ldg(g + q * sq + b * sb);
        }
#pragma unroll
        for (int s = 0; s < 2; s++) {
            long long re = fx::MIDDLE, im = fx::MIDDLE;
#pragma unroll
            for (int b = 0; b < 3; b++) {
                const int e = s * 3 + b;
                fx::mid_add(re, u[b].x, u[b].y, rh[e], rl[e]);
                fx::mid_add(re, sgn * u[b].z, sgn * u[b].w, ih[e], il[e]);
                fx::mid_add(im, u[b].x, u[b].y, ih[e], il[e]);
                fx::mid_add(im, -sgn * u[b].z, -sgn * u[b].w, rh[e], rl[e]);
            }
            fx::middle_done(re);
            fx::middle_done(im);
#pragma unroll
            for (int b = 0; b < 3; b++) {
                const int e = s * 3 + b;
                fx::wide_add(re, u[b].x, rh[e]);
                fx::wide_add(re, sgn * u[b].z, ih[e]);
                fx::wide_add(im, u[b].x, ih[e]);
                fx::wide_add(im, -sgn * u[b].z, rh[e]);
            }
            w[s * 3 + q].re = re;
            w[s * 3 + q].im = im;
            if (fx::guard_large(w[s * 3 + q].re, w[s * 3 + q].im)) large |= 1u << (s * 3 + q);
        }
    }
    // rebuild (w, sg B_mu^H w)
#pragma unroll
    for (int e = 0; e < 6; e++) acc[e] = add(acc[e], w[e]);
#define FX_REBUILD(F0, W0, F1, W1)                   \
    do {                                             \
        acc[6] = F0(acc[6], w[W0]);                  \
        acc[7] = F0(acc[7], w[W0 + 1]);              \
        acc[8] = F0(acc[8], w[W0 + 2]);              \
        acc[9] = F1(acc[9], w[W1]);                  \
        acc[10] = F1(acc[10], w[W1 + 1]);            \
        acc[11] = F1(acc[11], w[W1 + 2]);            \
    } while (0)
    switch (which) {
        case 0: FX_REBUILD(addi, 3, addi, 0); break;
        case 1: FX_REBUILD(subi, 3, subi, 0); break;
        case 2: FX_REBUILD(sub, 3, add, 0); break;
        case 3: FX_REBUILD(add, 3, sub, 0); break;
        case 4: FX_REBUILD(addi, 0, subi, 3); break;
        case 5: FX_REBUILD(subi, 0, addi, 3); break;
        case 6: FX_REBUILD(sub, 0, sub, 3); break;
        default: FX_REBUILD(add, 0, add, 3); break;
    }
#undef FX_REBUILD
}

// The elements g0 + i, i in todo, in FP64 and through the epilogue: two at a time, 16 lanes each.
// Returns what this lane's RHS gains in |result|^2.  prod: the warp's scratch.
template <bool DAG, int EPI>
__device__ __noinline__ double elements_fp64(const SplitArgs &a, unsigned todo, unsigned g0, Cx<double> (*prod)[8][2][3]) {
    const int lane = threadIdx.x & 31, grp = lane >> 4;
    const LaneRole role = lane_role<DAG>(lane & 15);
    double sum = 0.0;
    while (todo) {
        const int i0 = __ffs(todo) - 1;
        todo &= todo - 1;
        const int i1 = __ffs(todo) - 1;  // -1: none
        todo &= todo - 1;
        const int i = grp ? i1 : i0;
        const unsigned g = g0 + (i < 0 ? 0 : i);
        const double n = split_site<DAG, EPI>(a, role, i >= 0, g >> a.kshift, g & (a.k - 1), prod[grp]);
        if (EPI != SPL_PLAIN) {
            const double n0 = __shfl_sync(0xffffffffu, n, 0), n1 = __shfl_sync(0xffffffffu, n, 16);
            if (lane == i0) sum += n0;
            if (lane == i1) sum += n1;
        }
    }
    return sum;
}

template <bool DAG, int EPI>
__global__ void __launch_bounds__(FX_TPB, 4) k_dslash_fx(const __grid_constant__ FxArgs args) {
    __shared__ double smem[(FX_TPB / 32) * MAX_RHS];
    __shared__ Cx<double> prod[FX_TPB / 32][2][8][2][3];
    const SplitArgs &a = args.s;
    if (EPI == SPL_NORM || EPI == SPL_CG) {
        bool any = false;
        for (unsigned q = 0; q < a.k; q++) any = any || a.st[q].active;
        if (!any) return;
    }
    const unsigned total = a.V << a.kshift;
    const size_t P = total;
    const unsigned s1 = a.L0, s2 = a.L0 * a.L1, s3 = s2 * a.L2, lane = threadIdx.x & 31;
    double nrm = 0.0;
    // a warp's lanes make the same number of passes (elements_fp64 takes them all)
    for (unsigned g0 = blockIdx.x * FX_TPB + (threadIdx.x & ~31u); g0 < total; g0 += gridDim.x * FX_TPB) {
        const unsigned g = g0 + lane;
        bool fp64 = false;  // left to elements_fp64
        if (g < total) {
            const unsigned s = g >> a.kshift, r = g & (a.k - 1);
            unsigned x, y, z, t, sl;
            if (a.eo >= 0) {
                const unsigned rest = a.lh > 1 ? fastdiv(s, a.dh) : s, q2 = fastdiv(rest, a.d1);
                t = fastdiv(q2, a.d2);
                y = rest - q2 * a.L1;
                z = q2 - t * a.L2;
                x = 2 * (s - rest * a.lh) + ((a.eo + y + z + t) & 1);
                sl = x + rest * a.L0;
            } else {
                const unsigned q1 = fastdiv(s, a.d0), q2 = fastdiv(q1, a.d1);
                t = fastdiv(q2, a.d2);
                x = s - q1 * a.L0;
                y = q1 - q2 * a.L1;
                z = q2 - t * a.L2;
                sl = s;
            }
            // neighbour of hop h = 2 mu + (backward) as a lattice site
            auto neighbour = [&](int h) {
                const int mu = h >> 1;
                const unsigned c = mu == 0 ? x : (mu == 1 ? y : (mu == 2 ? z : t));
                const unsigned L = mu == 0 ? a.L0 : (mu == 1 ? a.L1 : (mu == 2 ? a.L2 : a.L3));
                const unsigned st = mu == 0 ? 1u : (mu == 1 ? s1 : (mu == 2 ? s2 : s3));
                return (h & 1) ? (c == 0 ? sl + (L - 1) * st : sl - st) : (c == L - 1 ? sl - (L - 1) * st : sl + st);
            };
            auto field_index = [&](unsigned nl) { return ((a.eo >= 0 ? nl >> 1 : nl) << a.kshift) + r; };
            int e[8], em = 1;
            unsigned sp0 = 0, sp1 = 0;  // nonzero spins of the neighbours in x and y, in z and t
#pragma unroll
            for (int h = 0; h < 8; h++) {
                const int w = __ldg(args.ex + field_index(neighbour(h)));
                e[h] = w & 0x7ff;
                em = max(em, e[h]);
                (h < 4 ? sp0 : sp1) |= (unsigned)w >> fx::NZ;
            }
            unsigned long long shifts = 0;  // alignment of each hop, 8 bits each
#pragma unroll
            for (int h = 0; h < 8; h++) shifts |= (unsigned long long)min(em - e[h], 63) << (8 * h);
            unsigned formed = fx::guard_formed(sp0, true) | (fx::guard_formed(sp1, false) << 8), large = 0;
            const int er = em + args.gscale;  // of the results
            fp64 = fx::exponent_bad(em, sp0 | sp1) || fx::exponent_bad(er, sp0 | sp1);
            if (!fp64) {
                I2 acc[12];
#pragma unroll
                for (int q = 0; q < 12; q++) acc[q].re = acc[q].im = 0;
                unsigned nl = neighbour(0);
#pragma unroll 1
                for (int h = 0; h < 8; h++) {
                    const bool bwd = h & 1;
                    // ask L1 for the next hop's data while this one is computed (the last hop asks for
                    // its own again: a branch cost more)
                    const unsigned nx = h < 7 ? neighbour(h + 1) : nl;
                    prefetch_hop_fx(args, ((h + 1) >> 1) & 3, field_index(nx), bwd ? sl : nx);
                    hop_fx(args, h >> 1, bwd, DAG != bwd, field_index(nl), bwd ? nl : sl, (int)(shifts & 63), acc, large);
                    shifts >>= 8;
                    nl = nx;
                    if (h == 3) large <<= 8;  // the x and y hops are done
                }
                fp64 = fx::guard_bad(formed & 63, large >> 8, formed >> 8, large & 63);
                if (!fp64) {
                    // diag * centre + hcoef * hops, then the epilogue, component by component
                    const double d = a.diag, hc = a.hcoef;
                    double al = 0.0;
                    if (EPI == SPL_CG) {
                        const CGScalars &st = a.st[r];
                        al = st.active ? st.alpha : 0.0;
                    }
                    const double2 *cen = static_cast<const double2 *>(a.cen);
                    double2 *res = static_cast<double2 *>(a.r);
                    double n2 = 0.0;
#pragma unroll
                    for (int q = 0; q < 12; q++) {
                        const size_t o = (size_t)q * P + g;
                        const double2 c0 = cen ? cen[o] : make_double2(0.0, 0.0);
                        double2 w = make_double2(d * c0.x + hc * fx::to_double(acc[q].re, er),
                                                 d * c0.y + hc * fx::to_double(acc[q].im, er));
                        if (EPI == SPL_PLAIN || EPI == SPL_NORM) {
                            static_cast<double2 *>(a.out)[o] = w;
                        } else if (EPI == SPL_CG) {
                            if (a.save_t) static_cast<double2 *>(a.tsave)[(size_t)q * a.V + s] = w;
                            double2 rr = res[o];
                            rr.x -= al * w.x;
                            rr.y -= al * w.y;
                            res[o] = rr;
                            w = rr;
                        } else {
                            const double2 bb = static_cast<const double2 *>(a.b)[o];
                            w = make_double2(bb.x - w.x, bb.y - w.y);
                            res[o] = w;
                        }
                        if (EPI != SPL_PLAIN) n2 += w.x * w.x + w.y * w.y;
                    }
                    nrm += n2;
                }
            }
        }
        __syncwarp();
        const unsigned todo = __ballot_sync(0xffffffffu, fp64);
        if (todo) nrm += elements_fp64<DAG, EPI>(a, todo, g0, prod[threadIdx.x >> 5]);
    }
    if (EPI == SPL_PLAIN) return;
    const double bs = block_reduce_rhs(nrm, (int)a.k, smem);
    const int k = (int)a.k;
    CGScalars *const sts = a.st;
    double *const h_alpha = a.h_alpha, *const h_beta = a.h_beta, *const h_rho = a.h_rho;
    const int iter = a.iter + (a.jbase ? *a.jbase : 0), set_rho = a.set_rho;
    grid_reduce_rhs(bs, k, a.partials, a.counter, smem, [=](int rr, double tot) {
        finish_scalars<EPI>(sts, h_alpha, h_beta, h_rho, iter, k, set_rho, rr, tot);
    });
}

template <int EPI>
cudaError_t fx_launch(bool dag, const FxArgs &a, int cap, cudaStream_t s) {
    const long n = (long)a.s.V << a.s.kshift;
    long grid = (n + FX_TPB - 1) / FX_TPB;
    const long most = (long)device_sm_count() * 4;  // resident blocks
    if (EPI != SPL_PLAIN && grid > most) grid = most;
    if (cap > 0 && grid > cap) grid = cap;
    if (dag) k_dslash_fx<true, EPI><<<(int)grid, FX_TPB, 0, s>>>(a);
    else k_dslash_fx<false, EPI><<<(int)grid, FX_TPB, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

// bytes of the integer field of n (site, RHS) pairs and of the links of V sites
size_t fx_field_bytes(long n) { return (size_t)((n + TILE - 1) / TILE) * TILE * 12 * 16; }
size_t fx_link_bytes(long V) { return 4 * fx_link_plane((unsigned)V) * 16; }

cudaError_t launch_links_range(const void *g64, long V, unsigned *range, cudaStream_t s) {
    ProfScope prof("links_range", (double)V * 4 * 144.0, s);
    long grid = (4 * V + 127) / 128;
    const long cap = (long)device_sm_count() * 16;
    if (grid > cap) grid = cap;
    cudaError_t e = cudaMemsetAsync(range, 0, sizeof(unsigned), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(range + 1, 0xff, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    k_links_range<<<(int)grid, 128, 0, s>>>(static_cast<const double2 *>(g64), (unsigned)V, range);
    return cudaGetLastError();
}

cudaError_t launch_links_fx(const void *g64, void *gfx, long V, int scale, cudaStream_t s) {
    ProfScope prof("links_fx", (double)V * 4 * 288.0, s);
    long grid = (4 * V + 127) / 128;
    const long cap = (long)device_sm_count() * 16;
    if (grid > cap) grid = cap;
    k_links_fx<<<(int)grid, 128, 0, s>>>(static_cast<const double2 *>(g64), static_cast<int4 *>(gfx), (unsigned)V,
                                         ldexp(1.0, 58 - scale));
    return cudaGetLastError();
}

cudaError_t launch_dslash_fx(const DslashCall &c, int epi, Field b, Field r, Field t_save, CGScalars *st, History h,
                             int iter, bool set_rho, RedScratch red, cudaStream_t s) {
    FxArgs a;
    split_args(a.s, c);
    if (c.eo_parity >= 0 && c.diag == 0.0) a.s.cen = nullptr;
    split_reduction(a.s, st, h, iter, red);
    a.s.r = r.v.data;
    a.s.b = b.v.data;
    a.s.tsave = t_save.v.data;
    a.s.save_t = t_save.v.data != nullptr;
    a.s.set_rho = set_rho;
    a.fx = static_cast<const longlong2 *>(c.fx.data);
    a.ex = c.fx.ex;
    a.g = static_cast<const int4 *>(c.fx.links);
    a.gscale = c.fx.scale;
    const unsigned n = a.s.V << a.s.kshift;
    {
        long grid = (n + FX_TPB - 1) / FX_TPB;
        k_to_fx<<<(int)grid, FX_TPB, 0, s>>>(static_cast<const double2 *>(c.in.v.data),
                                                static_cast<longlong2 *>(c.fx.data), c.fx.ex, n);
    }
    switch (epi) {
        case SPL_PLAIN: return fx_launch<SPL_PLAIN>(c.dagger, a, 0, s);
        case SPL_NORM: return fx_launch<SPL_NORM>(c.dagger, a, red.max_blocks, s);
        case SPL_CG: return fx_launch<SPL_CG>(c.dagger, a, red.max_blocks, s);
        default: return fx_launch<SPL_RESID>(c.dagger, a, red.max_blocks, s);
    }
}

}  // namespace eig
