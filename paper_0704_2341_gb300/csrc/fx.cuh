// Block fixed-point arithmetic for the FP64 Wilson stencil.
//
// GB300 retires 1.6 FP64 instructions per clock per SM (measured), but 25 integer
// multiply-adds 32 x 32 + 64 bit (a product and a 64-bit add), so the hop
// products are done in integers.  A site's 24 reals share one exponent: fixed =
// x 2^60 / 2^e with every |x| < 2^e, 61 significant bits for the largest component
// where a double has 53.  Links (-1/2 U) are fixed = u 2^61.  A 64 x 64 bit product
// is taken as a1 b1 + (a1 b0 + a0 b1) / 2^32 from signed 32-bit limbs (a = a1 2^32 +
// a0, a0 in [-2^31, 2^31)): three multiply-adds per real product.  The middle terms
// are summed over a row before they are rounded; a0 b0 (below one unit, zero mean)
// is dropped.  One unit of a hop sum is 2^-57 of the largest input component
// around the output site.  Against a 64-bit-mantissa reference of D x (8^4,
// Gaussian x) the relative error is 5.9e-17, of which rounding the result to
// double is 4.7e-17; the double-precision kernel, whose hop arithmetic rounds some
// sixty times at 2^-53 of its partial sums, is 9.3e-17 off.  That holds for vectors
// whose components are of like size; where one is small beside its neighbours its
// digits below the unit are lost, so wilson_apply sends such tiles to double
// precision (fx_weak, dslash_fx.cuh).
//
// Ranges: |u 2^61| <= 2^60 x 1.01, |x 2^60 / 2^e| < 2^60, a projected component
// h below 2^61.  A row's middle sum has six terms u.hi h.lo, below 2^60 |u| each, and
// six u.lo h.hi, below 2^60 each: with R = the sum of |re| + |im| over a row (forward hop)
// or a column (backward hop) of the link it stays below (R + 6) 2^60, so R <= kFxRowMax
// = 1.9 keeps it below 7.9 2^60 < 2^63.  (R is at most sqrt 6 / 2 = 1.23 for a unitary U; six entries
// at the limit of kFxLinkMax alone would reach 9.03 2^60.)  The row's products are then below
// 1.9 2^58, and eight hops below 2^62.  Entries and R are checked when the links are
// packed; a field that fails either check is done in double precision.
#pragma once

#include <stdint.h>

#include "gs_internal.cuh"

namespace gs {

constexpr int kFxZero = 0;        // exponent word of a site whose components are all zero
constexpr int kFxBad = -1;        // a component is not finite, or the site's scale is out of range
constexpr int kFxMinExp = 128, kFxMaxExp = 1920;   // accepted biased exponents of a site's largest component
constexpr double kFxLinkMax = 0.505;               // largest |re|, |im| of -1/2 U (0.5 for a unitary U)
constexpr double kFxRowMax = 1.9;                  // largest sum of |re| + |im| over a row or column of -1/2 U

struct FxLimb {
    int hi, lo;
};

__host__ __device__ __forceinline__ FxLimb fx_split(long long v) {
    const unsigned lo = (unsigned)v, hi = (unsigned)((unsigned long long)v >> 32);
    return FxLimb{(int)(hi + (lo >> 31)), (int)lo};
}

// Whether the three entries p[0], p[ld], p[2 ld] of a packed link, limbs (re.lo, re.hi,
// im.lo, im.hi), have a sum of |re| + |im| within kFxRowMax.
__host__ __device__ __forceinline__ bool fx_row_fits(const int4* p, int ld) {
    long long sum = 0;
    for (int c = 0; c < 3; ++c) {
        const int4 u = p[c * ld];
        const long long re = (long long)u.y * 4294967296ll + u.x, im = (long long)u.w * 4294967296ll + u.z;
        sum += (re < 0 ? -re : re) + (im < 0 ? -im : im);
    }
    return sum <= (long long)(kFxRowMax * 2305843009213693952.0);     // 2^61
}

// accumulator of products: hh counts 2^64 units, md 2^32 units
struct FxAcc {
    long long hh, md;
};

// s + a b as one 32 x 32 + 64 bit multiply-add (written out: from the C
// expression the compiler makes full 64 x 64 bit products)
__host__ __device__ __forceinline__ long long fx_mad(int a, int b, long long s) {
#ifdef __CUDA_ARCH__
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s) : "r"(a), "r"(b));
    return s;
#else
    return s + (long long)a * b;
#endif
}

__host__ __device__ __forceinline__ void fx_fma(FxAcc& s, FxLimb a, FxLimb b) {
    s.hh = fx_mad(a.hi, b.hi, s.hh);
    s.md = fx_mad(a.hi, b.lo, s.md);
    s.md = fx_mad(a.lo, b.hi, s.md);
}

// an accumulator whose value, after the rounding of the middle terms and a
// right shift by sh, is rounded to nearest
__host__ __device__ __forceinline__ FxAcc fx_start(long long half) {
    FxAcc s;
    s.hh = half;
    s.md = 0x80000000ll;
    return s;
}

__host__ __device__ __forceinline__ long long fx_take(const FxAcc& s, int sh) {
#ifdef __CUDA_ARCH__
    long long t;
    asm("{.reg .u32 a, b, c, d, e;\n\t"
        "mov.b64 {a, b}, %1;\n\t"
        "mov.b64 {c, d}, %2;\n\t"
        "shr.s32 e, d, 31;\n\t"
        "add.cc.u32 a, a, d;\n\t"
        "addc.u32 b, b, e;\n\t"
        "mov.b64 %0, {a, b};}"
        : "=l"(t) : "l"(s.hh), "l"(s.md));
    return t >> sh;
#else
    return (s.hh + (s.md >> 32)) >> sh;
#endif
}

// biased exponent of a double (0 for zeros and denormals, 2047 for Inf and NaN)
__host__ __device__ __forceinline__ int fx_exponent(unsigned hi) { return (int)((hi >> 20) & 0x7ffu); }

// x 2^60 / 2^(E - 1022), rounded, for a double of biased exponent at most E
// (denormals count as zero: they lie 2^76 below the smallest accepted site
// scale)
__host__ __device__ __forceinline__ long long fx_from_bits(unsigned hi, unsigned lo, int E) {
    const int ex = fx_exponent(hi);
    int sh = E - ex;
    sh = sh > 63 ? 63 : sh;
    unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    m = ((m << 7) + (sh > 0 ? 1ull << (sh - 1) : 0ull)) >> sh;
    if (ex == 0) m = 0;
    return (int)hi < 0 ? -(long long)m : (long long)m;
}

// S 2^(E - 1022 - 57) as a double, rounded to nearest even (E within the
// accepted range: the result is a normal double)
__host__ __device__ __forceinline__ double fx_to_double(long long S, int E) {
    if (S == 0) return 0.0;
    const unsigned long long u = S < 0 ? 0ull - (unsigned long long)S : (unsigned long long)S;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)u);
#else
    const int lz = __builtin_clzll(u);
#endif
    const unsigned long long m = u << lz;
    unsigned long long r = m >> 11;
    const unsigned tail = (unsigned)m & 0x7ffu;
    r += (tail + ((unsigned)r & 1u) > 0x400u) ? 1u : 0u;     // half rounds to even
    // r carries its leading one into the exponent field
    unsigned long long bits = ((unsigned long long)(unsigned)(E + 6 - lz) << 52) + r;
    if (S < 0) bits |= 0x8000000000000000ull;
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)bits);
#else
    double d;
    memcpy(&d, &bits, sizeof d);
    return d;
#endif
}

// Fixed-point arrays keep 32 sites together, component-major inside: entry
// (site, c) of a k-component array is at fx_index(site, k) + 32 c, so that the
// components of a site have constant offsets and those of consecutive sites
// share lines.
__host__ __device__ __forceinline__ int64_t fx_index(int site, int k) {
#ifdef __CUDA_ARCH__
    int64_t i;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(i) : "r"(site >> 5), "r"(32 * k));
    return i + (site & 31);
#else
    return (int64_t)(site >> 5) * (32 * k) + (site & 31);
#endif
}
constexpr int64_t fx_padded(int64_t sites) { return (sites + 31) / 32 * 32; }

}  // namespace gs
