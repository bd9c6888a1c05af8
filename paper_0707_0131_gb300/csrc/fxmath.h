// Block fixed-point arithmetic of the FP64-accurate stencil (dslash_fx.cu): conversions between
// FP64 and 64-bit integers with a shared exponent, and the 29-bit limbs of their products.
// Host and device code, so that it can be checked on the CPU.
//
// A number x with |x| < 2^(emax - 1022) (emax: the largest biased exponent of its block) is held
// as I = x 2^(1079 - emax), rounded, |I| <= 2^57.  Links (|u| <= 1) are held as u 2^58.  An
// integer I = hi 2^29 + lo is split into signed limbs (|lo| <= 2^28), and a product u I is formed
// in units of I as  hi hi + (hi lo + lo hi) 2^-29;  the dropped lo lo 2^-58 is at most 1/4 unit.
//
// Errors of one hop component w = sum over 3 colours of u (a +- b), in units of I (2^-57 of the
// next power of two above the largest component M of the eight neighbours), for links whose rows
// have norm 1:
//   inputs     to_fixed rounds a and b by 1/2 each, align shifts that and rounds a +- b by 1/2: at
//              most 1 per real of a +- b, and sqrt(6) < 2.5 over a row of norm 1
//   links      1/2 2^-58 on six |a +- b| <= 2^58: 3
//   products   1/4 each for lo lo: 1.5, and 1/2 for the rounding of the middle limb
// 7.5 units for any one hop, 60 for the sum of eight (the integer sums are exact), one FP64
// rounding at the end; random signs give 2 to 4 units.  60 units are 2^-50 M.
//
// An error relative to M is not one relative to a component: FP64 keeps a component that its
// neighbours' large ones never touch (other spins, or other colours where links do not mix them)
// to its own precision.  So an element keeps the fixed-point result only if every output component
// it forms is large enough (guard_bad): |re| or |im| of one of its x and y hop products, or of one
// of its z and t hop products, reaches 2^GUARD_BIT units, a sixteenth of the power of two above M.
// Then 60 units are below 60 times 2^-53 of the sum of the component's terms |u| |a +- b|; the
// FP64 chain's own bound is 15 times.  Simulated against exact sums over fields spread by site,
// spin, colour or component and point sources, with random, near-unit and unit links: the errors of
// kept elements are 0.7 to 3.9 times 2^-53 of those terms at most, the FP64 chain's 1.8 to 6.0, and
// smaller than that in each class (with alignment by floor up to 6.8, and larger in three).  Of
// Gaussian fields the guard leaves fewer than one element in 10^9 to FP64; twice the bound would
// leave one in 10^5, and one in 500 where a source has a single colour (16^3x32, k = 4, such a
// source: 8% over a dense one with this bound, 70% with twice it).
#pragma once
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace eig {
namespace fx {

constexpr int LIMB = 29;
constexpr int SPECIAL = 0x7ff;  // exponent of a block with an Inf or NaN

FX_HD uint64_t bits(double x) {
#if defined(__CUDA_ARCH__)
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
#endif
}
FX_HD double from_bits(uint64_t u) {
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)u);
#else
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}
FX_HD int clz64(uint64_t u) {
#if defined(__CUDA_ARCH__)
    return __clzll((long long)u);
#else
    return u ? __builtin_clzll(u) : 64;
#endif
}

// x 2^(1079 - emax) rounded to the nearest integer (ties away from zero)
FX_HD long long to_fixed(double x, int emax) {
    const uint64_t u = bits(x);
    const int e = (int)((u >> 52) & 0x7ff);
    uint64_t m = u & 0xfffffffffffffull;
    if (e) m |= 0x10000000000000ull;
    int d = emax - (e > 1 ? e : 1);
    if (d > 63) d = 63;
    m = ((m << 5) >> d) + 1 >> 1;
    const long long s = (long long)u >> 63;
    return ((long long)m ^ s) - s;
}

// a 2^(emax - 1079) rounded to the nearest double (ties away from zero; results below the
// normal range become zero)
FX_HD double to_double(long long a, int emax) {
    const long long s = a >> 63;
    const uint64_t m = (uint64_t)((a ^ s) - s);
    const int lz = clz64(m);
    const uint64_t A = m << (lz & 63);
    const uint64_t r = (A >> 11) + ((A >> 10) & 1);  // 2^52 .. 2^53
    int be = emax - lz + 7;
    uint64_t out = r + ((uint64_t)(be - 1) << 52);
    if (be >= 2047) out = 0x7ff0000000000000ull;
    if (be < 1 || m == 0) out = 0;
    return from_bits(out | ((uint64_t)s & 0x8000000000000000ull));
}

// I 2^-sh rounded to the nearest integer (ties up), 0 <= sh <= 63, |I| <= 2^58
FX_HD long long align(long long I, int sh) {
    return (long long)((uint64_t)I + ((1ull << sh) >> 1)) >> sh;
}

// I = hi 2^29 + lo, -2^28 <= lo < 2^28
FX_HD void limbs(long long I, int &hi, int &lo) {
    hi = (int)((I + (1ll << (LIMB - 1))) >> LIMB);
    lo = (int)((uint32_t)(uint64_t)I << (32 - LIMB)) >> (32 - LIMB);
}

// acc + a b, one wide multiply-add (written out: left to itself the compiler widens the limbs
// first and multiplies 64 by 64 bits, four instructions instead of one)
FX_HD void wide_add(long long &acc, int a, int b) {
#if defined(__CUDA_ARCH__)
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
#else
    acc += (long long)a * b;
#endif
}
// A sum of products u I in units of I: acc starts as MIDDLE (half a unit of the result), takes the hi lo
// + lo hi products (mid_add), is brought to units of I (middle_done), and takes the hi hi products
// (wide_add).  One accumulator in turn for both needs fewer registers and no addition at the end.
constexpr long long MIDDLE = 1ll << (LIMB - 1);
FX_HD void mid_add(long long &acc, int uh, int ul, int h, int l) {
    wide_add(acc, uh, l);
    wide_add(acc, ul, h);
}
FX_HD void middle_done(long long &acc) { acc >>= LIMB; }

// The power of two that links are held relative to: the largest squared norm of a row or column, as
// its high word top, then lies between 1/2 and 2 (a norm of sqrt 2 keeps the sums of eight hops below
// 2^63, and the bounds above grow by it).  False where the fixed-point form is not for these links:
// Inf or NaN, near the ends of the exponent range, all zero, or the smallest nonzero norm (bottom) less
// than 1/16 of the largest, where too many elements would fail the guard.
FX_HD bool link_scale(unsigned top, unsigned bottom, int &scale) {
    const int et = (int)(top >> 20) - 1022, eb = (int)(bottom >> 20) - 1022;  // norms^2 in [2^(e-1), 2^e)
    scale = et >= 1 ? et / 2 : -((1 - et) / 2);
    return top < 0x7fe00000u && et > -900 && et < 900 && et - eb <= 8;
}

// The guard.  Exponent words hold a block's exponent and, from bit NZ on, which of its four spins
// have a nonzero component.  Blocks whose largest exponent lies outside [EX_LOW, EX_HIGH) are left
// to FP64 too: results could be subnormal, or FP64 overflow where integers do not.
constexpr int NZ = 16;
constexpr int EX_LOW = 57, EX_HIGH = 2041;
constexpr int GUARD_BIT = 53;

FX_HD bool exponent_bad(int emax, unsigned spins) { return spins && (emax < EX_LOW || emax >= EX_HIGH); }

// whether a hop product is large enough for the guard (one unit off where negative)
FX_HD bool guard_large(long long re, long long im) {
    const int r = (int)(re >> 32), i = (int)(im >> 32);
    return ((unsigned)((r ^ (r >> 31)) | (i ^ (i >> 31))) >> (GUARD_BIT - 32)) != 0;
}

// which upper components (3 bits per half-spinor spin) hops of mu 0, 1 (xy) or 2, 3 form from
// anything but zeros, from the OR of their neighbours' spin bits
FX_HD unsigned guard_formed(unsigned spins, bool xy) {
    const unsigned part = xy ? ((spins >> 3) & 1) | ((spins >> 1) & 2) : spins >> 2;  // partners of spins 0, 1
    const unsigned u = (spins | part) & 3;
    return (u & 1 ? 7u : 0u) | (u & 2 ? 56u : 0u);
}

// formed0 / large0: of the hops of mu 0 and 1, formed1 / large1: of mu 2 and 3.  Upper component e
// sums product e of every hop; lower spins take the other spin's product from mu 0 and 1.
FX_HD bool guard_bad(unsigned formed0, unsigned large0, unsigned formed1, unsigned large1) {
    const unsigned f0x = ((formed0 & 7) << 3) | (formed0 >> 3), l0x = ((large0 & 7) << 3) | (large0 >> 3);
    return (((formed0 | formed1) & ~(large0 | large1)) | ((f0x | formed1) & ~(l0x | large1))) != 0;
}

}  // namespace fx
}  // namespace eig
