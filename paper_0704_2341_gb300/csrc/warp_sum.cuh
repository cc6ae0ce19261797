// Sums across a warp in integers, for code whose double-precision additions
// would be bound by the FP64 pipe (20 clocks of an SM per warp instruction).
#pragma once

#include "fx.cuh"

namespace gs {
namespace {

// Integer sum over the warp of m, |m| < 2^58, in every lane.
__device__ __forceinline__ long long warp_add(long long m) {
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)m & 0x1fffffu);
    const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(m >> 21) & 0x1fffffu);
    const int hi = __reduce_add_sync(0xffffffffu, (int)(m >> 42));
    return (long long)lo + ((long long)mid << 21) + ((long long)hi << 42);
}

// The sum over the warp of N <= 16 doubles per lane, in every lane.  Values are
// added as 54-bit integers under the largest one's exponent: a term is off by up to
// 2^-54 of the largest one, the sum exact but for that.  For terms of like size, as the
// threads' shares of a dot are, that is less than a double-precision tree loses,
// which rounds every partial sum at 2^-53; for uneven ones it is more.  Rms error of 320
// terms in units of the largest, integers / tree: Gaussian 4.5e-16 / 9.5e-16, Gaussian
// spread over six decades 4.3e-16 / 3.5e-16, one term a thousand times the rest
// 4.4e-16 / 1.6e-16.  Sums out of the usual range take that tree; with REFINE
// also sums that cancel to nothing, where it still has the small terms' last bits: a
// host-driven Krylov method takes an exact zero for a breakdown (one of 16 runs of
// 3000 steps that do not converge met rho = 0).  The persistent FP64 solver goes
// without it: its host takes a solve that ended on a zero again in double
// precision.
template <int N, bool REFINE = false>
__device__ __forceinline__ double warp_sum(const double (&x)[N]) {
    static_assert(N <= 16, "the integer sum would overflow");
    int E = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) E = max(E, fx_exponent((unsigned)__double2hiint(x[k])));
    E = __reduce_max_sync(0xffffffffu, E);
    if (E == 0) return 0.0;
    if (E >= kFxMinExp && E <= 1900) {
        long long m = 0;
#pragma unroll
        for (int k = 0; k < N; ++k)
            m += fx_from_bits((unsigned)__double2hiint(x[k]), (unsigned)__double2loint(x[k]), E + 6);
        m = warp_add(m);
        if (!REFINE || m != 0) return fx_to_double(m, E + 3);
    }
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < N; ++k) s += x[k];
#pragma unroll 1
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return s;
}

// The same for floats: 54 bits, of which 24 are the largest value's own; the small terms'
// bits below 2^-54 of it are cut off.
template <int N>
__device__ __forceinline__ double warp_sum(const float (&x)[N]) {
    static_assert(N <= 16, "the integer sum would overflow");
    unsigned E = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) E = max(E, (__float_as_uint(x[k]) >> 23) & 0xffu);
    E = __reduce_max_sync(0xffffffffu, E);
    if (E == 255u || E == 0u) {            // Inf, NaN, or nothing above the denormals
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < N; ++k) s += (double)x[k];
#pragma unroll 1
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        return s;
    }
    long long m = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const unsigned b = __float_as_uint(x[k]), e = (b >> 23) & 0xffu;
        const unsigned sh = min(E - max(e, 1u), 63u);
        const unsigned long long a = ((unsigned long long)((b & 0x7fffffu) | (e ? 0x800000u : 0u)) << 30) >> sh;
        m += (int)b < 0 ? -(long long)a : (long long)a;
    }
    // m counts 2^(E - 150 - 30); fx_to_double's unit is 2^(its exponent - 1079)
    return fx_to_double(warp_add(m), (int)E + 899);
}

}  // namespace
}  // namespace gs
