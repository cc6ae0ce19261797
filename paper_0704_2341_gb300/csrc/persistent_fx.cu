// Persistent FP64 BiCGStab on D_rr with the stencils in block fixed point: the
// whole inner solve in one cooperative launch, as k_bicg_persistent_f64
// (persistent.cu, which remains for fields and right-hand sides that fixed
// point cannot hold).
//
// What bounds an iteration on 8^4 (3840 rest sites, one tile of 26 sites on
// each of 148 SMs): the double-precision kernel spent 22 of its 46 us in the two
// stencils, at 1.6 FP64 instructions per clock per SM, and the rest in vector
// updates, four grid barriers and four reductions.  Here the stencils are
// integer work; the vector updates and the dot products stay double.
//   * A block owns its tiles' sites in every phase, a thread one complex
//     component of one site (warp = component, lane = site), so p and s in fixed
//     point are all that other blocks read.
//   * They are exchanged without a barrier or a fence: every 16-byte word carries
//     the parity of the iteration that wrote it in its lowest bit (2^-60 of the
//     site's largest component), the exponent's word the iteration itself, and
//     the thread that needs the site reads until they are right, one trip through
//     L2.  A site is overwritten only after a reduction that its readers joined
//     after reading.
//   * Two reductions an iteration: ||r||^2 of the updates travels with
//     <rhat, v>, and ||s||^2, <rhat, s> with t's sums.  Convergence is seen one
//     stencil later, with the same result.  A reduction is an exchange of
//     (value, epoch) words: a block publishes its sums, all blocks poll the
//     words themselves, and no counter is needed.
//   * An FP64 instruction occupies a quarter SM's pipe for 80 clocks.  Sums over
//     threads and blocks are therefore taken in integers (warp_sum), and the
//     update of x and the norms run beside the hops' integer work.
#include "dslash_fx.cuh"
#include "gridsync.cuh"
#include "warp_sum.cuh"

namespace gs {
namespace {

constexpr int kFxMaxGrid = 512;    // blocks of the cooperative grid
constexpr int kFxRec = 8;          // (value, epoch) words per block and parity: one 128-byte line
constexpr int kFxMark = 0xfff;     // exponent code of a site whose values are not finite or out of range

struct FxOut {                     // a vector as its neighbours read it
    longlong2* m;                  // mantissas (fx_index)
    unsigned* e;                   // iteration << 12 | exponent code (0: zero site, kFxMark)
};

struct PArgsFx {
    StencilArgs A, C;              // the D_rr stencils of p and of s (sets, links, fixed-point input)
    const double2* b;              // right-hand side, [site][12]
    double2* x;                    // solution, [site][12]
    FxOut p, s;
    double2 *r, *rhat, *v, *t, *xi, *pd, *sd;   // the solver's vectors (not RES)
    int64_t n;                     // sites
    int ts;                        // sites per tile (<= 32)
    double tol;
    int maxit;
    ulonglong2* rec;               // [2 parities][gridDim][kFxRec], epochs zeroed before the launch
    int* err;
    unsigned long long wait_ns;
    BicgState* st;
    unsigned long long* phases;    // [16] or null: cycles per phase (block 0)
};

// Kernel shapes.  RES: one tile a block, whose links (36 KB) and private vectors
// (42 KB) stay in shared memory for the whole solve; otherwise any number of
// tiles, with the vectors in memory.  NS = 1: 16 warps a block, one block an SM,
// the shortest iteration; NS = 2: 8 warps a block, two blocks an SM.
template <int NS>
constexpr int kT = kFxThreads<NS>;

template <int NS, bool RES>
struct FxSmem {
    union {
        FxShared hop;
        double part[8][kT<NS>];                  // a reduction's values by thread
        double tot[8][kFxMaxGrid];               // and by block
    };
    int sE[8][kSitesPerBlock];
    int sM[12][kSitesPerBlock];
    double blk[8];
    double sum[8];
    double2 sc[5];                 // alpha, omega, beta, rho, <rhat, v>
    int flag, far;                 // far: beta_far
    double2 vec[RES ? 7 : 1][RES ? 12 : 1][kSitesPerBlock];      // r, rhat, v, t, x, p, s
    int4 link[RES ? 8 : 1][RES ? 9 : 1][kSitesPerBlock];         // [hop][entry][site]
};


// A 16-byte word read or written whole.
__device__ __forceinline__ void rec_store(ulonglong2* p, unsigned long long v, unsigned long long e) {
    asm volatile("{.reg .b128 q; mov.b128 q, {%1, %2}; st.relaxed.gpu.global.b128 [%0], q;}" ::"l"(p), "l"(v), "l"(e)
                 : "memory");
}
__device__ __forceinline__ ulonglong2 rec_load(const ulonglong2* p) {
    ulonglong2 r;
    asm volatile("{.reg .b128 q; ld.relaxed.gpu.global.b128 q, [%2]; mov.b128 {%0, %1}, q;}"
                 : "=l"(r.x), "=l"(r.y) : "l"(p) : "memory");
    return r;
}

// A waiting thread's bound: false once the context's wait limit has passed or
// another thread of the grid has given up (asked every 64 polls).
__device__ __noinline__ bool fx_still(const PArgsFx& P, unsigned long long& t0, unsigned spins) {
    const unsigned long long now = global_ns();
    if (t0 == 0) t0 = now;
    if (vload(P.err) != 0) return false;
    if (now - t0 <= P.wait_ns && spins <= (unsigned)kSpinLimit) return true;
    atomicExch(P.err, (int)GS_TIMEOUT);
    return false;
}

// Grid barrier and sums in one: tot = the sums over all threads of the grid of
// v[q], the same bits in every block.  False (in every thread) if a wait ran
// out or another block gave up.  A block writes word k + 2 over word k only
// after every block has read word k (it has passed barrier k + 1, for which
// every block first finished barrier k).  Eight lanes read a block's line.
template <int NV, int NS, bool RES>
__device__ bool grid_reduce(const PArgsFx& P, FxSmem<NS, RES>& sm, unsigned& epoch, const double (&v)[NV], double (&tot)[NV]) {
    constexpr int T = kT<NS>, NW = T / 32;
    constexpr int LOG = NV > 4 ? 3 : NV > 2 ? 2 : NV > 1 ? 1 : 0;   // words read per block
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nb = gridDim.x;
    ++epoch;
    __syncthreads();               // the union's hop results have been read
#pragma unroll
    for (int q = 0; q < NV; ++q) sm.part[q][threadIdx.x] = v[q];
    __syncthreads();
    constexpr int used = NW < 12 ? NW : 12;      // warps that hold components
    for (int q = warp; q < NV; q += NW) {
        double x[used];
#pragma unroll
        for (int w = 0; w < used; ++w) x[w] = sm.part[q][w * 32 + lane];
        const double t = warp_sum<used>(x);
        if (lane == 0) sm.blk[q] = t;
    }
    __syncthreads();
    ulonglong2* rec = P.rec + (size_t)(epoch & 1) * nb * kFxRec;
    if (threadIdx.x < NV)
        rec_store(rec + (size_t)blockIdx.x * kFxRec + threadIdx.x,
                  (unsigned long long)__double_as_longlong(sm.blk[threadIdx.x]), epoch);
    bool ok = true;
    const int words = nb << LOG;
    for (int i0 = threadIdx.x; i0 < words && ok; i0 += 4 * T) {
        unsigned spins = 0;
        unsigned long long t0 = 0;
        int todo = 15;
        while (todo) {
            ulonglong2 w[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int i = i0 + m * T, q = i & ((1 << LOG) - 1);
                if (i >= words || q >= NV) todo &= ~(1 << m);
                else if (todo & (1 << m)) w[m] = rec_load(rec + (size_t)(i >> LOG) * kFxRec + q);
            }
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if ((todo & (1 << m)) && w[m].y == epoch) {
                    const int i = i0 + m * T;
                    sm.tot[i & ((1 << LOG) - 1)][i >> LOG] = __longlong_as_double((long long)w[m].x);
                    todo &= ~(1 << m);
                }
            if (todo && (++spins & 63) == 0 && !fx_still(P, t0, spins)) {
                ok = false;
                break;
            }
        }
    }
    if (!__syncthreads_and(ok)) return false;
    for (int q = warp; q < NV; q += NW) {
        constexpr int R = kFxMaxGrid / 32;
        double x[5], more[R - 5];
#pragma unroll
        for (int m = 0; m < 5; ++m) x[m] = lane + 32 * m < nb ? sm.tot[q][lane + 32 * m] : 0.0;
        double t = warp_sum<5>(x);
        if (nb > 160) {
#pragma unroll
            for (int m = 5; m < R; ++m) more[m - 5] = lane + 32 * m < nb ? sm.tot[q][lane + 32 * m] : 0.0;
            t += warp_sum<R - 5>(more);
        }
        if (lane == 0) sm.sum[q] = t;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) tot[q] = sm.sum[q];
    return true;
}

// The block's entries: calls f(site, component, index in the solver's vectors)
// for this thread's components of the tile at base.
template <int NS, bool RES, class F>
__device__ __forceinline__ void own_entries(const PArgsFx& P, int64_t base, F f) {
    const int lane = threadIdx.x & 31;
    const int64_t k = base + lane;
    if (lane >= P.ts || k >= P.n) return;
    const int64_t i = RES ? lane : fx_index((int)k, 12);
#pragma unroll 1
    for (int c = threadIdx.x >> 5; c < 12; c += kT<NS> / 32) f(k, c, i + 32 * c);
}

__device__ __forceinline__ int max_exponent(double2 v) {
    return max(fx_exponent((unsigned)__double2hiint(v.x)), fx_exponent((unsigned)__double2hiint(v.y)));
}

// Publishes a tile of u, whose entries' threads have just written d and put
// their exponents into sm.sM, in fixed point under the tag; returns the site's
// exponent.  Sites below the accepted scale count as zero (the right-hand side's
// own were checked: such a site is 2^-895 of the vector); a site with a value
// that is not finite, or beyond the scale, is marked and poisons its neighbours.
template <int NS, bool RES>
__device__ __forceinline__ int fx_publish(const PArgsFx& P, FxSmem<NS, RES>& sm, const FxOut& u, const double2* d,
                                          int64_t base, unsigned tag) {
    const int lane = threadIdx.x & 31;
    __syncthreads();
    int E = 0;
#pragma unroll
    for (int c = 0; c < 12; ++c) E = max(E, sm.sM[c][lane]);
    own_entries<NS, RES>(P, base, [&](int64_t k, int c, int64_t i) {
        const double2 v = d[i];
        const long long x = fx_from_bits((unsigned)__double2hiint(v.x), (unsigned)__double2loint(v.x), E);
        const long long y = fx_from_bits((unsigned)__double2hiint(v.y), (unsigned)__double2loint(v.y), E);
        rec_store((ulonglong2*)u.m + fx_index((int)k, 12) + 32 * c,
                  ((unsigned long long)x & ~1ull) | (unsigned long long)(tag & 1u), (unsigned long long)y);
        if (c == 0) {
            const unsigned code = E > kFxMaxExp ? (unsigned)kFxMark : E < kFxMinExp ? 0u : (unsigned)E;
            asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(u.e + k), "r"((tag << 12) | code) : "memory");
        }
    });
    return E;
}

// Input site i for hop w: reads until the site's words are of iteration tag.
// x = its exponent code; false if the wait ran out.
template <int NS>
__device__ __forceinline__ bool fx_fetch(const PArgsFx& P, const FxOut& u, int w, int i, unsigned tag, int& x,
                                         FxOperands<NS>& o) {
    const ulonglong2* p = (const ulonglong2*)u.m + fx_index(i, kSiteC);
    unsigned spins = 0;
    unsigned long long t0 = 0;
    for (;;) {
        unsigned word;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(word) : "l"(u.e + i) : "memory");
        unsigned stale = (word >> 12) ^ tag;
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const int s = (NS == 1 ? (w & 1) : k);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const ulonglong2 a = rec_load(p + (3 * s + c) * 32), b = rec_load(p + (fx_partner(w, s) + c) * 32);
                o.s[k][c] = make_longlong2((long long)a.x, (long long)a.y);
                o.q[k][c] = make_longlong2((long long)b.x, (long long)b.y);
                stale |= (((unsigned)a.x ^ tag) | ((unsigned)b.x ^ tag)) & 1u;
            }
        }
        x = (int)(word & 0xfffu);
        if (stale == 0) return true;
        if ((++spins & 63) == 0 && !fx_still(P, t0, spins)) return false;
    }
}

// out = D_rr u with the phase's dots added to e: DOTS = 2: <rhat, out>; 5: <out,
// s>, <out, out>, <rhat, out> (u = s).  beside(base) is double-precision work on
// the tile's own entries that runs beside the hops.  False in every thread if a
// wait ran out.
template <int DOTS, int NS, bool RES, int NE, class F>
__device__ __forceinline__ bool stencil_phase(const PArgsFx& P, const StencilArgs& a, FxSmem<NS, RES>& sm, const FxOut& u,
                                              unsigned tag, int l0, const double2* d, const double2* rhat, double2* out,
                                              double (&e)[NE], F beside) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = warp * NS;
    const int64_t step = (int64_t)gridDim.x * P.ts;
    int l = l0;
    for (int64_t base = (int64_t)blockIdx.x * P.ts; base < P.n; base += step) {
        const unsigned i = l < 0 ? 0xffffffffu : (unsigned)l - (unsigned)a.a0;
        int x = 0;
        bool ok = true;
        FxOperands<NS> o;
        if (i < (unsigned)P.n) {
            if (!RES) fx_load_link<NS>(a, w, (w & 2) ? l : (int)(a.o0 + base) + lane, o);
            ok = fx_fetch<NS>(P, u, w, (int)i, tag, x, o);
        }
        if (!RES && base + step < P.n) l = fx_label(a, base + step, P.ts, w);
        if (NS == 2 || !(w & 1)) sm.sE[w >> 1][lane] = x;
        if (!__syncthreads_and(ok)) return false;
        int E = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) E = max(E, sm.sE[q][lane]);
        beside(base);
        if (x > 0 && E - x < 63) {
            if (RES) {
                const int4(&L)[9][kSitesPerBlock] = *(const int4(*)[9][kSitesPerBlock])sm.link[RES ? w >> 1 : 0];
#pragma unroll
                for (int k = 0; k < 9; ++k) o.u[k] = L[k][lane];
            }
            fx_hop<NS>(o, w, E - x, sm.hop, lane);
        } else {
#pragma unroll
            for (int k = 0; k < NS; ++k)
#pragma unroll
                for (int q = 0; q < 3; ++q) sm.hop.hop[w + k][lane][q] = make_longlong2(0, 0);
        }
        __syncthreads();
        own_entries<NS, RES>(P, base, [&](int64_t, int c, int64_t i) {
            const double2 self = d[i], rv = rhat[i];
            const I2 h = fx_sum(sm.hop, lane, c / 3, c % 3);
            double re = fma(a.diag, self.x, fx_to_double(h.x, E));
            double im = fma(a.diag, self.y, fx_to_double(h.y, E));
            if (E == kFxMark) re = im = __longlong_as_double(0x7ff8000000000000ll);
            out[i] = make_double2(re, im);
            if constexpr (DOTS == 2) {
                e[0] = fma(rv.x, re, fma(rv.y, im, e[0]));
                e[1] = fma(rv.x, im, fma(-rv.y, re, e[1]));
            } else {
                e[0] = fma(re, self.x, fma(im, self.y, e[0]));
                e[1] = fma(re, self.y, fma(-im, self.x, e[1]));
                e[2] = fma(re, re, fma(im, im, e[2]));
                e[3] = fma(rv.x, re, fma(rv.y, im, e[3]));
                e[4] = fma(rv.x, im, fma(-rv.y, re, e[4]));
            }
        });
        __syncthreads();
    }
    return true;
}

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 zdiv(double2 a, double2 b) {
    const double inv = 1.0 / (b.x * b.x + b.y * b.y);
    return make_double2((a.x * b.x + a.y * b.y) * inv, (a.y * b.x - a.x * b.y) * inv);
}

// d 2^k exactly (zero below the normal numbers, infinite above them; not finite stays as it is)
__device__ __forceinline__ double shift2(double d, int k) {
    const int hi = __double2hiint(d), ex = fx_exponent((unsigned)hi);
    if (ex == 2047) return d;
    if (ex == 0 || ex + k <= 0) return 0.0;
    if (ex + k >= 2047) return hi < 0 ? -1.0 / 0.0 : 1.0 / 0.0;
    return __hiloint2double(hi + k * (1 << 20), __double2loint(d));
}
__device__ __forceinline__ double2 shift2(double2 v, int k) { return make_double2(shift2(v.x, k), shift2(v.y, k)); }

// beta = rho' tt / (rv ts).  The products grow with the eighth power of the right-hand
// side's norm: ||b|| = 1e40 made beta 0 and 1e-40 infinite.  Away from the middle of
// the range (beta_far) every number therefore goes in with its exponent taken out
// and the sum of the exponents comes back at the end.  Powers of two change no rounding.
__device__ __forceinline__ double2 beta_factor(double2 rv, double2 ts, double tt) {      // tt / (rv ts)
    const double x = fma(rv.x, ts.x, -(rv.y * ts.y)), y = fma(rv.x, ts.y, rv.y * ts.x);
    const double inv = 1.0 / fma(x, x, y * y);
    return make_double2(tt * x * inv, -(tt * y) * inv);
}
__device__ __forceinline__ double2 beta_product(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ bool beta_far(double2 rv, double2 ts, double tt) {
    constexpr int mid = 1023, near = 240;
    const int et = fx_exponent((unsigned)__double2hiint(tt));
    return max(max(abs(max_exponent(rv) - mid), abs(max_exponent(ts) - mid)), abs(et - mid)) > near;
}
__device__ __noinline__ double2 beta_far_out(double2 rho, double2 rv, double2 ts, double tt) {
    const int er = max_exponent(rv) - 1023, es = max_exponent(ts) - 1023, e = max_exponent(rho) - 1023;
    const int et = fx_exponent((unsigned)__double2hiint(tt)) - 1023;
    return shift2(beta_product(shift2(rho, -e), beta_factor(shift2(rv, -er), shift2(ts, -es), shift2(tt, -et))),
                  e + et - er - es);
}

struct FxClock {   // phase clock of block 0 (profiling only)
    unsigned long long* out;
    long long t;
    __device__ void start(unsigned long long* p) {
        out = (blockIdx.x == 0 && threadIdx.x == 0) ? p : nullptr;
        t = out ? clock64() : 0;
    }
    __device__ __forceinline__ void mark(int i) {
        if (out) {
            const long long now = clock64();
            out[i] += (unsigned long long)(now - t);
            t = now;
        }
    }
};

// The recurrence is that of k_bicg_persistent_f64: A (v = D p), B (s = r - alpha
// v), C (t = D s), D (x, r and p).
template <int NS, bool RES>
__global__ void __launch_bounds__(kT<NS>, NS) k_bicg_persistent_fx(const __grid_constant__ PArgsFx P) {
    extern __shared__ __align__(16) unsigned char dyn[];
    FxSmem<NS, RES>& sm = *(FxSmem<NS, RES>*)dyn;
    double2* const mine = &sm.vec[0][0][0];
    constexpr int kVec = 12 * kSitesPerBlock;
    double2* const r = RES ? mine : P.r;
    double2* const rhat = RES ? mine + kVec : P.rhat;
    double2* const vv = RES ? mine + 2 * kVec : P.v;
    double2* const tt = RES ? mine + 3 * kVec : P.t;
    double2* const xx = RES ? mine + 4 * kVec : P.xi;
    double2* const pd = RES ? mine + 5 * kVec : P.pd;
    double2* const sd = RES ? mine + 6 * kVec : P.sd;
    const int lane = threadIdx.x & 31;
    const int64_t step = (int64_t)gridDim.x * P.ts, first = (int64_t)blockIdx.x * P.ts;
    unsigned epoch = 0;
    int iter = 0, status = GS_OK;
    bool ok, conv = false, early = false;
    double rr, bb, tol2;
    {   // x = 0, r = rhat = p = b, ||b||^2, and whether b and the links fit
        double v[2] = {0.0, 0.0};
        for (int64_t base = first; base < P.n; base += step) {
            own_entries<NS, RES>(P, base, [&](int64_t k, int c, int64_t i) {
                const double2 b = __ldg(P.b + k * 12 + c);
                xx[i] = make_double2(0.0, 0.0);
                r[i] = rhat[i] = pd[i] = b;
                v[0] = fma(b.x, b.x, fma(b.y, b.y, v[0]));
                sm.sM[c][lane] = max_exponent(b);
            });
            int E = fx_publish<NS, RES>(P, sm, P.p, pd, base, 1u);
            if (lane >= P.ts || base + lane >= P.n) E = kFxMinExp;
            if (E > kFxMaxExp || (E > 0 && E < kFxMinExp)) v[1] = 1.0;
            else if (E == 0)
                own_entries<NS, RES>(P, base, [&](int64_t, int, int64_t i) {
                    if (r[i].x != 0.0 || r[i].y != 0.0) v[1] = 1.0;   // denormals only
                });
            __syncthreads();
        }
        if (__ldg(P.A.fxflag) != 0) v[1] = 1.0;
        double tot[2];
        ok = grid_reduce<2, NS, RES>(P, sm, epoch, v, tot);
        bb = rr = ok ? tot[0] : 0.0;
        tol2 = P.tol * P.tol * bb;
        if (ok && tot[1] != 0.0) status = kFxUnfit;
        else if (ok && !(bb > 0.0)) {
            conv = (bb == 0.0);
            if (!conv) status = GS_NONFINITE;
        }
        if (threadIdx.x == 0) sm.sc[3] = make_double2(bb, 0.0);
        __syncthreads();
    }
    // the updates of x and ||r||^2 that phase D leaves for the next phase A
    double vr = 0.0;          // this thread's part of ||r||^2
    auto finish_updates = [&](int64_t base) {
        const double2 al = sm.sc[0], om = sm.sc[1];
        own_entries<NS, RES>(P, base, [&](int64_t, int, int64_t i) {
            const double2 pi = tt[i], si = sd[i], ri = r[i];     // p before its update
            double2 xi = xx[i];
            xi.x = fma(al.x, pi.x, fma(-al.y, pi.y, xi.x));
            xi.y = fma(al.x, pi.y, fma(al.y, pi.x, xi.y));
            xi.x = fma(om.x, si.x, fma(-om.y, si.y, xi.x));
            xi.y = fma(om.x, si.y, fma(om.y, si.x, xi.y));
            xx[i] = xi;
            vr = fma(ri.x, ri.x, fma(ri.y, ri.y, vr));
        });
    };
    const int l0 = fx_label(P.A, first, P.ts, (threadIdx.x >> 5) * NS);
    bool pending = false;     // a breakdown unless that residual shows convergence
    // the state after the updates: false once the solve has ended
    auto judge = [&](double r2) {
        rr = r2;
        if (!isfinite(rr)) status = GS_NONFINITE;
        else if (rr <= tol2) conv = true;
        else if (pending) status = GS_BREAKDOWN;
        return !conv && status == GS_OK;
    };
    if (RES && l0 >= 0 && (NS == 2 || !((threadIdx.x >> 5) & 1))) {     // this hop's link of the tile's site
        const int w = (threadIdx.x >> 5) * NS;
        FxOperands<1> o;
        fx_load_link<1>(P.A, w, (w & 2) ? l0 : (int)(P.A.o0 + first) + lane, o);
#pragma unroll
        for (int q = 0; q < 9; ++q) sm.link[RES ? w >> 1 : 0][RES ? q : 0][lane] = o.u[q];
    }
    __syncthreads();
    FxClock pc;
    pc.start(P.phases);
    while (ok && !conv && status == GS_OK && iter < P.maxit) {
        const unsigned tag = (unsigned)(iter + 1) & 0xfffffu;
        {   // A: v = D p, <rhat, v> -> alpha; ||r||^2
            double e[3] = {0.0, 0.0, 0.0}, tot[3];
            vr = 0.0;
            if (!(ok = stencil_phase<2, NS, RES>(P, P.A, sm, P.p, tag, l0, pd, rhat, vv, e, [&](int64_t base) {
                      if (iter > 0) finish_updates(base);
                  })))
                break;
            e[2] = vr;
            pc.mark(0);
            if (!(ok = grid_reduce<3, NS, RES>(P, sm, epoch, e, tot))) break;
            pc.mark(1);
            if (iter > 0 && !judge(tot[2])) break;
            if (threadIdx.x == 0) {
                int f = 0;
                if (tot[0] == 0.0 && tot[1] == 0.0) f = 10 + GS_BREAKDOWN;
                else {
                    const double2 al = zdiv(sm.sc[3], make_double2(tot[0], tot[1]));
                    sm.sc[0] = al;
                    sm.sc[4] = make_double2(tot[0], tot[1]);
                    if (!isfinite(al.x) || !isfinite(al.y)) f = 10 + GS_NONFINITE;
                }
                sm.flag = f;
            }
            __syncthreads();
            pc.mark(2);
            if (sm.flag >= 10) {
                status = sm.flag - 10;
                break;
            }
        }
        // B: s = r - alpha v
        double e[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0}, tot[8];
        {
            const double2 al = sm.sc[0];
            for (int64_t base = first; base < P.n; base += step) {
                own_entries<NS, RES>(P, base, [&](int64_t, int c, int64_t i) {
                    const double2 vi = vv[i], ri = r[i];
                    double2 si;
                    si.x = ri.x - (al.x * vi.x - al.y * vi.y);
                    si.y = ri.y - (al.x * vi.y + al.y * vi.x);
                    sd[i] = si;
                    sm.sM[c][lane] = max_exponent(si);
                });
                fx_publish<NS, RES>(P, sm, P.s, sd, base, tag);
                if (base + step < P.n) __syncthreads();
            }
            pc.mark(3);
        }
        {   // C: t = D s, <t, s>, <t, t>, <rhat, t>, ||s||^2, <rhat, s> -> omega, rho', beta
            if (!(ok = stencil_phase<5, NS, RES>(P, P.C, sm, P.s, tag, l0, sd, rhat, tt, e, [&](int64_t base) {
                      own_entries<NS, RES>(P, base, [&](int64_t, int, int64_t i) {
                          const double2 si = sd[i], hi = rhat[i];
                          e[5] = fma(si.x, si.x, fma(si.y, si.y, e[5]));
                          e[6] = fma(hi.x, si.x, fma(hi.y, si.y, e[6]));
                          e[7] = fma(hi.x, si.y, fma(-hi.y, si.x, e[7]));
                      });
                  })))
                break;
            pc.mark(6);
            if (!(ok = grid_reduce<8, NS, RES>(P, sm, epoch, e, tot))) break;
            pc.mark(7);
            if (!isfinite(tot[5])) {
                status = GS_NONFINITE;
                break;
            }
            if (tot[5] <= tol2) {   // ||s||^2: x += alpha p below, after the loop
                rr = tot[5];
                ++iter;
                conv = early = true;
                break;
            }
            // Serial FP64 algebra: a step takes 0.05 us, so two warps on two
            // quarters of the SM share it (and a third looks at the range).  beta = (rho' / rho) (alpha / omega)
            // = rho' <t, t> / (<rhat, v> <t, s>).
            if (threadIdx.x == 0) {
                const double inv = tot[2] > 0.0 ? 1.0 / tot[2] : 0.0;
                const double2 om = make_double2(tot[0] * inv, tot[1] * inv);
                sm.sc[1] = om;
                sm.sc[3] = make_double2(tot[6] - (om.x * tot[3] - om.y * tot[4]),
                                        tot[7] - (om.x * tot[4] + om.y * tot[3]));
            } else if (threadIdx.x == 32) {
                sm.sc[2] = beta_factor(sm.sc[4], make_double2(tot[0], tot[1]), tot[2]);
            } else if (threadIdx.x == 64) {
                sm.far = beta_far(sm.sc[4], make_double2(tot[0], tot[1]), tot[2]);
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                const double2 om = sm.sc[1], rho_new = sm.sc[3];
                int f = (isfinite(om.x) && isfinite(om.y)) ? 0 : 10 + GS_NONFINITE;
                if (f == 0 && !(om.x == 0.0 && om.y == 0.0) && !(rho_new.x == 0.0 && rho_new.y == 0.0)) {
                    const double2 be = sm.far ? beta_far_out(rho_new, sm.sc[4], make_double2(tot[0], tot[1]), tot[2])
                                              : beta_product(rho_new, sm.sc[2]);
                    sm.sc[2] = be;
                    if (!isfinite(be.x) || !isfinite(be.y)) f = 10 + GS_NONFINITE;
                } else if (f == 0) {
                    f = 1;     // breakdown pending
                    sm.sc[2] = make_double2(0.0, 0.0);
                }
                sm.flag = f;
            }
            __syncthreads();
            pc.mark(8);
            if (sm.flag >= 10) {
                status = sm.flag - 10;
                break;
            }
        }
        {   // D: r = s - omega t ; p = r + beta (p - omega v)   (x += alpha p + omega s, ||r||^2: finish_updates)
            const double2 om = sm.sc[1], be = sm.sc[2];
            pending = sm.flag == 1;
            for (int64_t base = first; base < P.n; base += step) {
                own_entries<NS, RES>(P, base, [&](int64_t, int c, int64_t i) {
                    const double2 si = sd[i], ti = tt[i], vi = vv[i];
                    double2 pi = pd[i];
                    double2 ri;
                    ri.x = si.x - (om.x * ti.x - om.y * ti.y);
                    ri.y = si.y - (om.x * ti.y + om.y * ti.x);
                    r[i] = ri;
                    tt[i] = pi;
                    double2 z;
                    z.x = pi.x - (om.x * vi.x - om.y * vi.y);
                    z.y = pi.y - (om.x * vi.y + om.y * vi.x);
                    pi.x = fma(be.x, z.x, fma(-be.y, z.y, ri.x));
                    pi.y = fma(be.x, z.y, fma(be.y, z.x, ri.y));
                    pd[i] = pi;
                    sm.sM[c][lane] = max_exponent(pi);
                });
                fx_publish<NS, RES>(P, sm, P.p, pd, base, (unsigned)(iter + 2) & 0xfffffu);
                if (base + step < P.n) __syncthreads();
            }
            ++iter;
            pc.mark(9);
        }
        if (iter >= P.maxit) {     // the last residual has no stencil to travel with
            vr = 0.0;
            for (int64_t base = first; base < P.n; base += step) finish_updates(base);
            double v[1] = {vr}, t[1];
            if ((ok = grid_reduce<1, NS, RES>(P, sm, epoch, v, t))) judge(t[0]);
            break;
        }
    }
    // x in the caller's layout; converged on s: x += alpha p first
    if (status != kFxUnfit) {
        const double2 al = early ? sm.sc[0] : make_double2(0.0, 0.0);
        for (int64_t base = first; base < P.n; base += step)
            own_entries<NS, RES>(P, base, [&](int64_t k, int c, int64_t i) {
                double2 xi = xx[i];
                if (early) {
                    const double2 pi = pd[i];
                    xi.x = fma(al.x, pi.x, fma(-al.y, pi.y, xi.x));
                    xi.y = fma(al.x, pi.y, fma(al.y, pi.x, xi.y));
                }
                P.x[k * 12 + c] = xi;
            });
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        BicgState* st = P.st;
        st->iter = iter;
        st->rr = rr;
        st->bb = bb;
        st->status = ok ? status : (int)GS_TIMEOUT;
        st->done = (conv || !ok || status != GS_OK) ? 1 : 0;
        publish(st);
    }
}

}  // namespace

// device memory of the kernel besides the inner workspace
struct FxScratch {
    int64_t cap = 0;               // sites
    longlong2* m = nullptr;        // mantissas of p and of s
    int64_t vec_cap = 0;           // sites of x and r, which the on-chip form does without
    double2 *x = nullptr, *r = nullptr;   // r: the right-hand side may be the inner workspace's own r
    unsigned* e = nullptr;         // exponent words of p and of s
    ulonglong2* rec = nullptr;
    int* err = nullptr;
};

void free_persist_fx(gs_ctx* c) {
    FxScratch* f = (FxScratch*)c->persist_fx;
    if (!f) return;
    void* bufs[] = {f->m, f->x, f->r, f->e, f->rec, f->err};
    for (void* b : bufs) cudaFree(b);
    delete f;
    c->persist_fx = nullptr;
}

static gs_status fx_scratch(gs_ctx* c, int64_t sites, bool vectors, FxScratch** out) {
    FxScratch* f = (FxScratch*)c->persist_fx;
    if (f && f->cap < sites) {
        free_persist_fx(c);
        f = nullptr;
    }
    if (!f) {
        f = new FxScratch();
        c->persist_fx = f;
        const size_t vec = (size_t)fx_padded(sites) * kSiteC * 16;
        if (cudaMalloc(&f->m, 2 * vec) != cudaSuccess ||
            cudaMalloc(&f->e, 2 * sites * sizeof(unsigned)) != cudaSuccess ||
            cudaMalloc(&f->rec, 2 * kFxMaxGrid * kFxRec * sizeof(ulonglong2)) != cudaSuccess ||
            cudaMalloc(&f->err, sizeof(int)) != cudaSuccess) {
            cudaGetLastError();
            free_persist_fx(c);
            return set_err(c, GS_ENOMEM, "allocating the persistent solver's vectors failed");
        }
        f->cap = sites;
    }
    if (vectors && f->vec_cap < sites) {
        const size_t vec = (size_t)fx_padded(sites) * kSiteC * sizeof(double2);
        cudaFree(f->x);
        cudaFree(f->r);
        f->x = f->r = nullptr;
        f->vec_cap = 0;
        if (cudaMalloc(&f->x, vec) != cudaSuccess || cudaMalloc(&f->r, vec) != cudaSuccess) {
            cudaGetLastError();
            free_persist_fx(c);
            return set_err(c, GS_ENOMEM, "allocating the persistent solver's vectors failed");
        }
        f->vec_cap = sites;
    }
    *out = f;
    return GS_OK;
}

template <int NS, bool RES>
static gs_status launch_fx_solver(gs_ctx* c, PArgsFx& P, const FxScratch* f) {
    int per_sm = 0;
    auto kern = k_bicg_persistent_fx<NS, RES>;
    const int smem = (int)sizeof(FxSmem<NS, RES>);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kT<NS>, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return set_err(c, GS_ECUDA, "no co-resident grid for the persistent solver");
    }
    const int64_t tiles = (P.n + kSitesPerBlock - 1) / kSitesPerBlock;
    int64_t g = (int64_t)per_sm * c->num_sms;
    if (c->coop_block_cap > 0) {
        // GS_OPT_COOP_BLOCKS counts thirds of an SM, two blocks here take what three of
        // the double-precision solver's did: counts that fit the GPU together still do
        const int64_t cap = (int64_t)c->coop_block_cap * 2 / 3;
        if (g > cap) g = cap > 0 ? cap : 1;
    } else if (c->ledger) {
        const int64_t usable = ledger_capacity(per_sm, c->num_sms);
        const int64_t n = c->ledger->running.load() > 1 ? c->ledger->running.load() : 1;
        const int64_t share = RES ? tiles : usable / n;
        g = ledger_grant(c, usable, tiles, share > 0 ? share : 1, RES ? tiles : 1);
        if (g < 1) return set_err(c, GS_ECUDA, "no co-resident grid for the persistent solver");
    }
    if (g > P.n) g = P.n;
    if (g > kFxMaxGrid) g = kFxMaxGrid;
    // tiles of up to 32 sites that share the set evenly (3840 sites on 152
    // blocks: 26 per tile)
    const int64_t rounds = (P.n + g * kSitesPerBlock - 1) / (g * kSitesPerBlock);
    if (RES && rounds > 1) return set_err(c, GS_ECUDA, "the persistent solver's grid does not cover the set");
    P.ts = (int)((P.n + g * rounds - 1) / (g * rounds));
    g = (P.n + P.ts - 1) / P.ts < g ? (P.n + P.ts - 1) / P.ts : g;
    GS_CUDA(c, cudaMemsetAsync(f->rec, 0, 2 * (size_t)g * kFxRec * sizeof(ulonglong2), c->stream));
    GS_CUDA(c, cudaMemsetAsync(f->err, 0, sizeof(int), c->stream));
    // no iteration's tag: the first has tag 1
    GS_CUDA(c, cudaMemsetAsync(f->e, 0, 2 * (size_t)P.n * sizeof(unsigned), c->stream));
    GS_CUDA(c, cudaMemsetAsync(f->m, 0, 2 * (size_t)fx_padded(P.n) * kSiteC * sizeof(longlong2), c->stream));
    void* args[] = {&P};
    GS_CUDA(c, cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)g), dim3(kT<NS>), args, smem, c->stream));
    c->launches++;
    return GS_OK;
}

// Solves D_rr x = b (S: the D_rr stencil of the plan's rest set); the status
// kFxUnfit in w's published state means that fixed point cannot hold the
// problem and nothing was done.
gs_status persistent_bicg_fx(gs_ctx* c, const Plan* p, const StencilArgs& S, const double2* b, double2* x,
                             InnerWork& w, double tol, int maxit) {
    const int64_t n = S.n_out;
    // A set with a tile for every SM at most keeps everything on chip; in a
    // batched call of such sets only, with 8 warps a tile, so that two solves
    // share an SM.
    const bool small = c->coop_block_cap == 0 && n <= (int64_t)kSitesPerBlock * c->num_sms &&
                       (!c->ledger || c->ledger->resident);
    FxScratch* f = nullptr;
    gs_status s = fx_scratch(c, n, !small, &f);
    if (s != GS_OK) return s;
    PArgsFx P;
    memset(&P, 0, sizeof P);
    P.A = P.C = S;
    longlong2* sm = f->m + fx_padded(n) * kSiteC;
    fx_args(p, f->m, nullptr, n, &P.A);
    fx_args(p, sm, nullptr, n, &P.C);
    P.b = b;
    P.x = x;
    P.p = FxOut{f->m, f->e};
    P.s = FxOut{sm, f->e + n};
    P.pd = w.p;
    P.sd = w.s;
    P.r = f->r;
    P.rhat = w.rhat;
    P.v = w.v;
    P.t = w.t;
    P.xi = f->x;
    P.n = n;
    P.tol = tol;
    P.maxit = maxit;
    P.rec = f->rec;
    P.err = f->err;
    P.wait_ns = c->wait_ns ? c->wait_ns : kWaitNs;
    P.st = w.st;
    P.phases = c->prof.on ? c->prof.phases_dev : nullptr;
    if (!small) return launch_fx_solver<2, false>(c, P, f);
    return c->ledger ? launch_fx_solver<2, true>(c, P, f) : launch_fx_solver<1, true>(c, P, f);
}

}  // namespace gs
