// Device code of the Wilson stencil in block fixed point (fx.cuh): a block of 16
// warps computes a tile of up to 32 output sites.  The double-precision tile
// (dslash_f64.cuh) takes over for a tile whose inputs fixed point cannot hold.
#pragma once

#include "dslash_f64.cuh"
#include "fx.cuh"

namespace gs {
namespace {

// NS = spin components of the two-spinor per thread: 1 (16 warps a tile, the
// shortest tile) or 2 (8 warps, fewer instructions a site)
template <int NS>
constexpr int kFxThreads = 512 / NS;
constexpr int kFxRow = 3;   // complex numbers in a site's row of a hop component (odd: free of bank conflicts)

union FxShared {
    longlong2 hop[16][kSitesPerBlock][kFxRow];   // [4 mu + 2 backward + two-spinor component][site][colour]
    double f64[4][24][kSitesPerBlock];
};

struct I2 {  // re, im
    long long x, y;
};
__device__ __forceinline__ I2 operator+(I2 a, I2 b) { return I2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ I2 operator-(I2 a, I2 b) { return I2{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ I2 fx_add_i(I2 a, I2 b) { return I2{a.x - b.y, a.y + b.x}; }   // a + i b
__device__ __forceinline__ I2 fx_sub_i(I2 a, I2 b) { return I2{a.x + b.y, a.y - b.x}; }   // a - i b

// A thread's share of a hop: NS spin components of the projected two-spinor h =
// psi_up -+ X_mu psi_lo of one input site, times the link, in units of
// 2^(E - 1022 - 57); sh = E - the input site's exponent.  Stored is g = U h for a
// forward hop and conj(g), g = U^dag h, for a backward one: with h conjugated as
// well the backward product is U^T conj(h), so one piece of code serves all warps
// and the SM shares its instruction lines (eight specialised copies starved on
// instruction fetch).  Only the projection and the order of the link's entries
// branch on the hop w = 4 mu + 2 backward + first component.
template <int NS>
struct FxOperands {
    int4 u[9];                      // [c][r]: U for the forward hop, its transpose for the backward one
    longlong2 s[NS][3], q[NS][3];   // upper spin components and their partners among the lower ones
};

// X_mu pairs spins 0, 1 with 3, 2 (mu < 2) or 2, 3
__device__ __forceinline__ int fx_partner(int w, int s) { return ((w < 8) != (s != 0)) ? 9 : 6; }

// Mantissas and exponents are plain loads: the kernel that writes them may still be
// running when this one starts (programmatic launch), so they are not constant
// for this kernel's lifetime, as __ldg would have it, and only a plain load stays
// behind griddepcontrol.wait.
template <int NS>
__device__ __forceinline__ void fx_load_spinor(const StencilArgs& a, int w, int in, FxOperands<NS>& o) {
    const longlong2* p = a.fxm + fx_index(in, kSiteC);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const int s = (NS == 1 ? (w & 1) : k);
        const longlong2* ps = p + s * (3 * 32);
        const longlong2* pq = p + fx_partner(w, s) * 32;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            o.s[k][c] = ps[c * 32];
            o.q[k][c] = pq[c * 32];
        }
    }
}

template <int NS>
__device__ __forceinline__ void fx_load_link(const StencilArgs& a, int w, int jl, FxOperands<NS>& o) {
    const int4* L = a.fxl + fx_index(jl, 36) + (w >> 2) * (9 * 32);
    if (w & 2) {
#pragma unroll
        for (int k = 0; k < 9; ++k) o.u[k] = __ldg(L + k * 32);
    } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) o.u[3 * (k % 3) + k / 3] = __ldg(L + k * 32);
    }
}

// h (forward) or conj(h) (backward) of component c
__device__ __forceinline__ void fx_project(int w, const longlong2 (&s)[3], const longlong2 (&q)[3], I2 (&h)[3]) {
#define GS_FX_PROJECT(X, Y)                                              \
    _Pragma("unroll") for (int c = 0; c < 3; ++c) h[c] = I2{X, Y};       \
    break;
    switch (w) {
        case 0: case 1: case 8: GS_FX_PROJECT(s[c].x + q[c].y, s[c].y - q[c].x)        // s - i q
        case 9: GS_FX_PROJECT(s[c].x - q[c].y, s[c].y + q[c].x)                        // s + i q
        case 5: case 12: case 13: GS_FX_PROJECT(s[c].x - q[c].x, s[c].y - q[c].y)      // s - q
        case 4: GS_FX_PROJECT(s[c].x + q[c].x, s[c].y + q[c].y)                        // s + q
        case 2: case 3: case 10: GS_FX_PROJECT(s[c].x - q[c].y, -s[c].y - q[c].x)      // conj(s + i q)
        case 11: GS_FX_PROJECT(s[c].x + q[c].y, q[c].x - s[c].y)                       // conj(s - i q)
        case 6: GS_FX_PROJECT(s[c].x - q[c].x, q[c].y - s[c].y)                        // conj(s - q)
        default: GS_FX_PROJECT(s[c].x + q[c].x, -s[c].y - q[c].y)                      // conj(s + q)
    }
#undef GS_FX_PROJECT
}

template <int NS>
__device__ __forceinline__ void fx_hop(const FxOperands<NS>& o, int w, int sh, FxShared& sm, int lane) {
    FxLimb hx[NS][3], hy[NS][3], hn[NS][3];
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        I2 h[3];
        fx_project(w + k, o.s[k], o.q[k], h);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            hx[k][c] = fx_split(h[c].x);
            hy[k][c] = fx_split(h[c].y);
            hn[k][c] = fx_split(-h[c].y);
        }
    }
    const long long half = sh > 0 ? 1ll << (sh - 1) : 0ll;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            FxAcc re = fx_start(half), im = fx_start(half);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int4 u = o.u[3 * c + r];
                const FxLimb ux{u.y, u.x}, uy{u.w, u.z};
                fx_fma(re, ux, hx[k][c]);
                fx_fma(re, uy, hn[k][c]);
                fx_fma(im, ux, hy[k][c]);
                fx_fma(im, uy, hx[k][c]);
            }
            sm.hop[w + k][lane][r] = make_longlong2(fx_take(re, sh), fx_take(im, sh));
        }
}

// Epilogue dots of one complex output (see f64_tile).
template <int EPI>
__device__ __forceinline__ void stencil_dots(const StencilArgs& a, int64_t i, double re, double im, double (&e)[5]) {
    if (EPI == EPI_DOT_RHAT_V) {
        const double2 rv = a.epi_vec[i];
        e[0] = fma(rv.x, re, fma(rv.y, im, e[0]));
        e[1] = fma(rv.x, im, fma(-rv.y, re, e[1]));
    } else if (EPI == EPI_DOT_TS) {
        const double2 sv = a.epi_vec[i];
        e[0] = fma(re, sv.x, fma(im, sv.y, e[0]));
        e[1] = fma(re, sv.y, fma(-im, sv.x, e[1]));
        e[2] = fma(re, re, fma(im, im, e[2]));
    }
}

// The hops' contributions to one component of a site, spin = 0..3, colour c:
// upper spins add g, lower spins X_mu^dag (g_back - g_fwd); backward rows hold
// conj(g).
__device__ __forceinline__ I2 fx_sum(const FxShared& sm, int site, int spin, int c) {
    if (spin < 2) {
        I2 t[4];
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            const longlong2 f = sm.hop[4 * mu + spin][site][c], b = sm.hop[4 * mu + 2 + spin][site][c];
            t[mu] = I2{f.x + b.x, f.y - b.y};
        }
        return (t[0] + t[1]) + (t[2] + t[3]);
    }
    const int s = spin - 2;
    I2 d[4];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        const int w = 4 * mu + (mu < 2 ? 1 - s : s);
        const longlong2 f = sm.hop[w][site][c], b = sm.hop[w + 2][site][c];
        d[mu] = I2{b.x - f.x, -b.y - f.y};
    }
    if (s == 0) return fx_sub_i(fx_sub_i(d[1] + d[3], d[0]), d[2]);   // -i d0 + d1 - i d2 + d3
    return fx_add_i(fx_sub_i(d[3] - d[1], d[0]), d[2]);               // -i d0 - d1 + i d2 + d3
}

// Fixed point resolves 2^-57 of the largest input component around a site, double
// precision 2^-53 of the terms of each component: a component whose terms are all
// small beside that maximum (a weak spin component; a weak colour where the links
// are near the identity) would lose digits that double precision keeps.  Such a
// component is `weak`: every hop's contribution is below 2^-k of the scale 2^E, k by
// the number of hops in range, and its tile is done in double precision.  A tile
// in double precision takes some 15 us, so the lines lie where Gaussian spinors
// meet them in less than 1e-8 of the components: |re| and |im| of a contribution are
// both below 2^-8 with probability 3e-4, 2^-10 2e-5, 2^-16 5e-9.
// Contributions that are zero because their inputs are (point sources, single spin
// components) are exact in fixed point, which fx_tile checks.  Gaussian input: 8^4
// 8.2 us, 24^3 x 48 0.50 ms, as without all this; point source on 8^4 10.3 us; one spin
// component alone 12.3 us and 0.70 ms, beside others 1e-12 of it 20.5 us and 1.8 ms
// (every tile twice; in double precision alone 12.3 us and 1.03 ms).
constexpr int kFxWeak1 = 16, kFxWeak2 = 10, kFxWeak = 8;     // k for one hop, two, more

__device__ __forceinline__ int fx_weak_bits(int hops) {
    return 57 - (hops > 2 ? kFxWeak : hops > 1 ? kFxWeak2 : kFxWeak1);
}
// bits 32.. of the magnitude
__device__ __forceinline__ int fx_top(long long v) {
    const int hi = (int)(v >> 32);
    return hi ^ (hi >> 31);
}
constexpr int kFxWeakSum = 1 << (57 - kFxWeak + 3 - 32);     // a sum of up to eight such contributions stays below

// The label of the tile's site `lane`'s neighbour that hop w reads (-1: no such
// site); fetched a tile ahead of its use.
__device__ __forceinline__ int fx_label(const StencilArgs& a, int64_t base, int ts, int w) {
    const int64_t k = base + (threadIdx.x & 31);
    if ((int)(threadIdx.x & 31) >= ts || k >= a.n_out) return -1;
    const int2 n = __ldg(a.nbr + (a.o0 + k) * 4 + (w >> 2));
    return (w & 2) ? n.y : n.x;
}

// Exponent word of the input site with label l (kFxZero outside the input
// range) and its index.
__device__ __forceinline__ int fx_site(const StencilArgs& a, int l, unsigned& i) {
    i = l < 0 ? 0xffffffffu : (unsigned)l - (unsigned)a.a0;   // labels below the range wrap above it
    if (i >= (unsigned)a.fxn) return kFxZero;
    return a.fxe[i];
}

__device__ __forceinline__ bool fx_weak(const FxShared& sm, const int (&sE)[8][kSitesPerBlock], int site, int spin,
                                        int c) {
    int hops = 0, top = 0;
    const int w01 = spin < 2 ? spin : 3 - spin, w23 = spin & 1;      // row within a direction: mu < 2, mu >= 2
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const longlong2 g = sm.hop[2 * q + (q < 4 ? w01 : w23)][site][c];
        top |= fx_top(g.x) | fx_top(g.y);
        hops += sE[q][site] > 0;
    }
    return hops > 0 && top < 1 << (fx_weak_bits(hops) - 32);
}

// One tile of up to 32 output sites from base, l = fx_label of this tile.
// Phase 1: a warp per hop (and spin component).  Phase 2: three warps per spin
// component, a thread one complex output: sum of the hops, conversion,
// diagonal, addend and the epilogue dots.  Returns true if the tile has to be done
// in double precision: an input site does not fit fixed point (nothing is written), or
// with KEEP a component is weak.  The output is not the addend.
template <int EPI, int NS, bool KEEP>
__device__ __forceinline__ bool fx_tile(const StencilArgs& a, int64_t base, int l, FxShared& sm,
                                        int (&sE)[8][kSitesPerBlock], double (&e)[5]) {
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int w = warp * NS;
    bool bad;
    {
        unsigned i;
        const int x = fx_site(a, l, i);
        FxOperands<NS> o;
        if (i < (unsigned)a.fxn) {
            fx_load_spinor<NS>(a, w, (int)i, o);
            fx_load_link<NS>(a, w, (w & 2) ? l : (int)(a.o0 + base) + lane, o);
        }
        bad = x < 0;
        if (NS == 2 || !(w & 1)) sE[w >> 1][lane] = x;
        __syncthreads();
        int E = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) E = max(E, sE[q][lane]);
        if (x > 0 && E - x < 63) {
            fx_hop<NS>(o, w, E - x, sm, lane);
        } else {
#pragma unroll
            for (int k = 0; k < NS; ++k)
#pragma unroll
                for (int q = 0; q < 3; ++q) sm.hop[w + k][lane][q] = make_longlong2(0, 0);
        }
    }
    if (__syncthreads_or(bad)) return true;
    unsigned weak = 0;         // bit per component of this thread
    for (int v = warp; v < 12; v += kFxThreads<NS> / 32) {
        const int spin = v / 3;
        const int i = (v - 3 * spin) * 32 + lane;
        const int site = i / 3, c = i - 3 * site;
        if (base + site >= a.n_out) continue;
        const I2 t = fx_sum(sm, site, spin, c);
        int E = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) E = max(E, sE[q][site]);
        const int64_t j = a.o0 + base + site;
        if (KEEP && (fx_top(t.x) | fx_top(t.y)) < kFxWeakSum && fx_weak(sm, sE, site, spin, c)) weak |= 1u << v;
        const int k = 3 * spin + c;
        const double2* self = nullptr;
        if (j >= a.a0 && j < a.a1) self = a.inA + (j - a.a0) * kSiteC + k;
        else if (j >= a.a1 && j < a.b1) self = a.inB + (j - a.a1) * kSiteC + k;
        const int64_t o = (base + site) * kSiteC + k;
        double re = fx_to_double(t.x, E), im = fx_to_double(t.y, E);
        if (self) {
            const double2 sv = __ldg(self);
            re = fma(a.diag, sv.x, re);
            im = fma(a.diag, sv.y, im);
        }
        if (a.negate) {
            re = -re;
            im = -im;
        }
        if (a.addend) {
            const double2 av = a.addend[o];
            re += av.x;
            im += av.y;
        }
        a.out[o] = make_double2(re, im);
        stencil_dots<EPI>(a, o, re, im, e);
    }
    if (KEEP) {
        if (!__syncthreads_or(weak)) return false;
        // A component is weak for nothing if its inputs are zero (what fixed point gives,
        // zero, is then exact): every warp looks at the inputs of its hop.
        int(&live)[4][kSitesPerBlock] = *(int(*)[4][kSitesPerBlock])sm.hop;
        if (threadIdx.x < 4 * kSitesPerBlock) live[warp][lane] = 0;
        __syncthreads();
        if (sE[w >> 1][lane] > 0) {
            const double2* p = l < a.a1 ? a.inA + (int64_t)(l - (int)a.a0) * kSiteC : a.inB + (int64_t)(l - (int)a.a1) * kSiteC;
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                const int up = NS == 1 ? (w & 1) : k, lo = w < 8 ? 3 - up : 2 + up;
                bool any = false;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const double2 u = __ldg(p + 3 * up + c), v = __ldg(p + 3 * lo + c);
                    any |= u.x != 0.0 || u.y != 0.0 || v.x != 0.0 || v.y != 0.0;
                }
                if (any) live[up][lane] = live[lo][lane] = 1;
            }
        }
        __syncthreads();
        bool keep = false;
#pragma unroll 1
        for (int v = warp; v < 12; v += kFxThreads<NS> / 32)
            if (weak >> v & 1u) keep |= live[v / 3][((v % 3) * 32 + lane) / 3] != 0;
        return __syncthreads_or(keep);
    }
    __syncthreads();
    return false;
}

// Tiles of a block that double precision has to do, a bit each (V < 2^31 / 12 sites in
// tiles of 32 over 2 blocks an SM: at most 18 400 tiles a block on 152 SMs).
constexpr int kFxRedoWords = 640;

// The block's tiles of the stencil; those that fixed point cannot hold (all of
// them when a link does not fit) are done in double precision afterwards, so
// that the rare path costs the common one no registers.  With KEEP `redo` holds them, as
// the hops' sums are gone by then.
template <int EPI, int NS, bool KEEP>
__device__ __forceinline__ void fx_stencil(const StencilArgs& a, bool links_bad, FxShared& sm,
                                           int (&sE)[8][kSitesPerBlock], unsigned* redo, int l, double (&e)[5]) {
    const int64_t step = (int64_t)gridDim.x * kSitesPerBlock;
    const int w = (threadIdx.x >> 5) * NS;
    bool any = links_bad;
    if constexpr (KEEP) {
        for (int i = threadIdx.x; i < kFxRedoWords; i += kFxThreads<NS>) redo[i] = links_bad ? ~0u : 0u;
        int tile = 0;
        if (!links_bad)
            for (int64_t base = (int64_t)blockIdx.x * kSitesPerBlock; base < a.n_out; base += step, ++tile) {
                const int next = fx_label(a, base + step, kSitesPerBlock, w);
                if (fx_tile<EPI, NS, true>(a, base, l, sm, sE, e)) {
                    any = true;
                    if (threadIdx.x == 0) redo[tile >> 5] |= 1u << (tile & 31);
                }
                l = next;
            }
        if (any) {
            __syncthreads();
            tile = 0;
            for (int64_t base = (int64_t)blockIdx.x * kSitesPerBlock; base < a.n_out; base += step, ++tile)
                if (redo[tile >> 5] >> (tile & 31) & 1u) f64_tile<EPI>(a, base, kSitesPerBlock, sm.f64, e);
        }
        return;
    }
    if (!links_bad)
        for (int64_t base = (int64_t)blockIdx.x * kSitesPerBlock; base < a.n_out; base += step) {
            const int next = fx_label(a, base + step, kSitesPerBlock, w);
            any |= fx_tile<EPI, NS, false>(a, base, l, sm, sE, e);
            l = next;
        }
    if (any)
        for (int64_t base = (int64_t)blockIdx.x * kSitesPerBlock; base < a.n_out; base += step) {
            unsigned i;
            const bool bad = fx_site(a, fx_label(a, base, kSitesPerBlock, w), i) < 0;
            if (__syncthreads_or(bad) || links_bad) f64_tile<EPI>(a, base, kSitesPerBlock, sm.f64, e);
        }
}

}  // namespace
}  // namespace gs
