// Block fixed-point arithmetic of the FP64-accurate stencil (dslash_fx.cu): conversions between
// FP64 and 64-bit integers with a shared exponent, and the 29-bit limbs of their products.
// Host and device code, so that it can be checked on the CPU.
//
// A number x with |x| < 2^(emax - 1022) (emax: the largest biased exponent of its block) is held
// as I = x 2^(1079 - emax), rounded, |I| <= 2^57.  Links (|u| <= 1) are held as u 2^58.  An
// integer I = hi 2^29 + lo is split into signed limbs (|lo| <= 2^28), and a product u I is formed
// in units of I as  hi hi + (hi lo + lo hi) 2^-29;  the dropped lo lo 2^-58 is below 1/4 unit.
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

// I = hi 2^29 + lo, -2^28 <= lo < 2^28
FX_HD void limbs(long long I, int &hi, int &lo) {
    hi = (int)((I + (1ll << (LIMB - 1))) >> LIMB);
    lo = (int)((uint32_t)(uint64_t)I << (32 - LIMB)) >> (32 - LIMB);
}

// the sums of hi hi and of hi lo + lo hi products, and their value in units of I
struct Acc {
    long long hh, mid;
};
// acc + a b, one wide multiply-add (written out: left to itself the compiler widens the limbs
// first and multiplies 64 by 64 bits, four instructions instead of one)
FX_HD void wide_add(long long &acc, int a, int b) {
#if defined(__CUDA_ARCH__)
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
#else
    acc += (long long)a * b;
#endif
}
FX_HD void mul_add(Acc &a, int uh, int ul, int h, int l) {
    wide_add(a.hh, uh, h);
    wide_add(a.mid, uh, l);
    wide_add(a.mid, ul, h);
}
FX_HD long long value(long long hh, long long mid) { return hh + ((mid + (1ll << (LIMB - 1))) >> LIMB); }

}  // namespace fx
}  // namespace eig
