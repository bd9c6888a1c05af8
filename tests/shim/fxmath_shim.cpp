// Host build of the fixed-point arithmetic of the FP64 stencil (fxmath.h) for the CPU tests: the
// hop sum of one element as k_dslash_fx forms it, its guard, and the same sum in _Float128.
#include <algorithm>
#include <cmath>

#include "../../paper_0707_0131_gb300/csrc/fxmath.h"

using namespace eig;
typedef _Float128 Q;

extern "C" long long fx_to_fixed(double x, int e) { return fx::to_fixed(x, e); }
extern "C" double fx_to_double(long long a, int e) { return fx::to_double(a, e); }
extern "C" long long fx_align(long long a, int sh) { return fx::align(a, sh); }
extern "C" int fx_link_scale(double top, double bottom, int *scale) {  // squared norms
    return fx::link_scale((unsigned)(fx::bits(top) >> 32), (unsigned)(fx::bits(bottom) >> 32), *scale);
}
extern "C" long long fx_limbs(long long a) {  // hi 2^29 + lo, or a value far off if lo is out of range
    int hi, lo;
    fx::limbs(a, hi, lo);
    return lo < -(1 << 28) || lo >= (1 << 28) ? 1ll << 62 : (long long)hi * (1ll << 29) + lo;
}

// scale: the power of two the links are held relative to.
// psi: neighbours [8][12] complex, hop 2 mu + (backward); u: their links [8][3][3] complex;
// forward projectors I - g_mu, backward I + g_mu.  err: largest error of a component over 2^-53
// times the sum of its terms |u_ab| |h_b|; units: largest error in units of the integers, the final
// FP64 rounding taken off.  Returns 1 if the guard keeps the fixed-point result.
extern "C" int fx_element(const double *psi, const double *u, int scale, double *err, double *units) {
    static const int part[4][2] = {{1, 0}, {1, 0}, {0, 1}, {0, 1}};
    static const int fre[4][2] = {{0, 0}, {-1, 1}, {0, 0}, {1, 1}}, fim[4][2] = {{1, 1}, {0, 0}, {1, -1}, {0, 0}};
    int ex[8], em = 1;
    unsigned sp0 = 0, sp1 = 0;
    for (int h = 0; h < 8; h++) {
        ex[h] = 1;
        for (int q = 0; q < 24; q++) {
            const double x = psi[h * 24 + q];
            ex[h] = std::max(ex[h], (int)((fx::bits(x) >> 52) & 0x7ff));
            if (x != 0) (h < 4 ? sp0 : sp1) |= 1u << (q / 6);
        }
        em = std::max(em, ex[h]);
    }
    long long acc[12][2] = {};
    Q exact[12][2] = {}, terms[12] = {};
    unsigned large = 0;
    for (int h = 0; h < 8; h++) {
        const int mu = h >> 1, sg = (h & 1) ? 1 : -1, sh = std::min(em - ex[h], 63);
        const double *v = psi + h * 24, *g = u + h * 18;
        long long H[6][2], W[6][2];
        Q hq[6][2], wq[6][2], t[6];
        auto in = [&](int e, int c) { return fx::to_fixed(v[2 * e + c], ex[h]); };
        for (int s = 0; s < 2; s++)
            for (int c = 0; c < 3; c++) {
                const int e = 3 * s + c, p = 6 + 3 * part[mu][s] + c, fr = sg * fre[mu][s], fi = sg * fim[mu][s];
                H[e][0] = fx::align(in(e, 0) + fr * in(p, 0) - fi * in(p, 1), sh);
                H[e][1] = fx::align(in(e, 1) + fr * in(p, 1) + fi * in(p, 0), sh);
                hq[e][0] = (Q)v[2 * e] + fr * (Q)v[2 * p] - fi * (Q)v[2 * p + 1];
                hq[e][1] = (Q)v[2 * e + 1] + fr * (Q)v[2 * p + 1] + fi * (Q)v[2 * p];
            }
        for (int s = 0; s < 2; s++)
            for (int q = 0; q < 3; q++) {
                long long re = fx::MIDDLE, im = fx::MIDDLE;
                int ah[3], bh[3], rh[3], ih[3];
                const int w = 3 * s + q;
                wq[w][0] = wq[w][1] = t[w] = 0;
                for (int b = 0; b < 3; b++) {
                    const int e = 3 * s + b, l = (h & 1) ? 3 * b + q : 3 * q + b;
                    const double ur = g[2 * l], ui = (h & 1) ? -g[2 * l + 1] : g[2 * l + 1];
                    int al, bl, rl, il;
                    fx::limbs(std::llrint(ur * std::ldexp(1.0, 58 - scale)), ah[b], al);
                    fx::limbs(std::llrint(ui * std::ldexp(1.0, 58 - scale)), bh[b], bl);
                    fx::limbs(H[e][0], rh[b], rl);
                    fx::limbs(H[e][1], ih[b], il);
                    fx::mid_add(re, ah[b], al, rh[b], rl);
                    fx::mid_add(re, -bh[b], -bl, ih[b], il);
                    fx::mid_add(im, ah[b], al, ih[b], il);
                    fx::mid_add(im, bh[b], bl, rh[b], rl);
                    wq[w][0] += (Q)ur * hq[e][0] - (Q)ui * hq[e][1];
                    wq[w][1] += (Q)ur * hq[e][1] + (Q)ui * hq[e][0];
                    t[w] += (Q)(std::hypot(ur, ui) * std::hypot((double)hq[e][0], (double)hq[e][1]));
                }
                fx::middle_done(re);
                fx::middle_done(im);
                for (int b = 0; b < 3; b++) {
                    fx::wide_add(re, ah[b], rh[b]);
                    fx::wide_add(re, -bh[b], ih[b]);
                    fx::wide_add(im, ah[b], ih[b]);
                    fx::wide_add(im, bh[b], rh[b]);
                }
                W[w][0] = re;
                W[w][1] = im;
                if (fx::guard_large(W[w][0], W[w][1])) large |= 1u << w;
            }
        if (h == 3) large <<= 8;
        for (int e = 0; e < 12; e++) {
            const int s = e / 3, c = e % 3, w = s < 2 ? e : 3 * part[mu][s - 2] + c;
            const int fr = s < 2 ? 1 : sg * fre[mu][part[mu][s - 2]], fi = s < 2 ? 0 : -sg * fim[mu][part[mu][s - 2]];
            acc[e][0] += fr * W[w][0] - fi * W[w][1];
            acc[e][1] += fr * W[w][1] + fi * W[w][0];
            exact[e][0] += fr * wq[w][0] - fi * wq[w][1];
            exact[e][1] += fr * wq[w][1] + fi * wq[w][0];
            terms[e] += t[w];
        }
    }
    *err = *units = 0;
    const Q unit = (Q)std::ldexp(1.0, em + scale - 1079 + 500) * (Q)0x1p-500;
    for (int e = 0; e < 12; e++)
        for (int c = 0; c < 2; c++) {
            Q d = (Q)fx::to_double(acc[e][c], em + scale) - exact[e][c], a = exact[e][c];
            d = d < 0 ? -d : d;
            a = a < 0 ? -a : a;
            if (terms[e] > 0) *err = std::max(*err, (double)(d / terms[e]) * 0x1p53);
            else if (d > 0) *err = INFINITY;
            *units = std::max(*units, (double)((d - a * (Q)0x1p-53) / unit));
        }
    return !fx::exponent_bad(em, sp0 | sp1) && !fx::exponent_bad(em + scale, sp0 | sp1) &&
           !fx::guard_bad(fx::guard_formed(sp0, true), large >> 8, fx::guard_formed(sp1, false), large & 63);
}
