// The C -> C layer of the learned preconditioner (C = 24) on the fifth-generation
// tensor cores: tcgen05.mma (kind::f16, BF16 operands, FP32 accumulator in
// tensor memory), weights moved by the bulk-copy engine, neighbour
// activations gathered by cp.async and transported by the CTA's threads.
//
// The layer  out(x)[R, a] = sum_d sum_k W_d[R, k] (U_d(x) in(x + d))[k, a]
// is a real GEMM over rows p = 3 x + a (site, colour):
//   A[p, k'] = Re / Im of T_d(x)[k, a],  T_d(x) = U_d(x) in(x + d)
//   B[n', k'] = the real form of W_d:  out_re = W_re T_re - W_im T_im,
//               out_im = W_im T_re + W_re T_im
// with n' = 2 R + (re, im), k' = (d, quarter, 2 kk + (re, im)), k = 24 quarter + kk.
// M = 256 rows per tile (two 128-lane accumulators), N = 192, K = 9 x 192,
// taken in 36 chunks of 48 (one transport, 24 input rows).  Operands are in
// the no-swizzle K-major core-matrix layout: an 8-row x 16-byte core matrix
// is 128 contiguous bytes, core matrices adjacent in K are 128 bytes apart
// (leading byte offset), 8-row groups 768 bytes apart (stride byte offset).
// The input activations are BF16 ([V][96][3] complex as bf16x2).
//
// Warp roles.  A tile is 85 sites (255 of the 256 GEMM rows) in 11 groups of
// 8; warps 0-10 own a group each, so a warp depends on no other until the
// tensor core: at chunk j it gathers its sites' raw rows of chunk j + 3 by
// cp.async (four raw buffers), transports chunk j into the A stage (two
// stages, reused once the tensor core has committed the chunk two back) and
// arrives on the stage's full barrier.  Warp 11 moves B_j by a bulk copy and
// issues the chunk's six MMAs as soon as the stage is full, then commits them
// to the stage's done barrier.  Every wait is bounded (the context's wait
// limit, GS_OPT_WAIT_LIMIT_US, 1 s by default); on a timeout the kernel
// stops, waits (bounded) for the MMAs it committed, frees its tensor memory
// and raises err.
//
// Bound by the transport's instructions: 36 multiply-adds a row and hop,
// against 7.3 % of the time in the tensor core at its peak.  With the rows of
// a site spread over 15 warps a (row, site) item took 172 warp instructions
// (index arithmetic, links reloaded, gather loop) and a block barrier a chunk
// left the schedulers idle half the time.  Here a lane keeps its site's link in
// registers for a transport's four chunks, each component twice, and two rows
// share every multiply-add (fma.rn.f32x2).  16^3 x 32 under the profiler: 1.11 ms
// -> 0.60 ms.
#include <cuda_bf16.h>
#include <stdint.h>

#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kRows = 256;                       // GEMM rows per tile
constexpr int kTileSites = 85;                   // sites per tile (row 255 is not used)
constexpr int kRC = 96;                          // 4 C, C = 24
constexpr int kN = 192;                          // real output columns
constexpr int kQ = 24;                           // input rows per chunk
constexpr int kKC = 2 * kQ;                      // real K per chunk
constexpr int kChunks = 36;                      // 9 transports x 4 quarters
constexpr int kStageWarps = 11;                  // gather + transport, 8 sites each; warp 11 issues B and the MMAs
constexpr int kThreads = 32 * (kStageWarps + 1);
constexpr int kSites = 8 * kStageWarps;          // site slots of a tile
constexpr int kRaw = 4;                          // raw buffers
constexpr int kPieces = 8 * 18;                  // 16-byte pieces of a warp's raw rows of a chunk
constexpr uint32_t kSBO = (kKC / 8) * 128;       // 768
constexpr uint32_t kABytes = kRows * kKC * 2;    // 24576
constexpr uint32_t kBBytes = kN * kKC * 2;       // 18432
constexpr uint32_t kPStride = kQ * 3 * 4 + 16;   // 304: raw rows of one site (+16 against bank conflicts)
constexpr uint32_t kPBytes = kSites * kPStride;  // 26752
constexpr uint32_t kUBytes = kSites * 9 * 8;     // 6336
// dynamic shared memory map (offsets from a 128-byte aligned base): A and B
// stages x 2, raw rows x 4, links x 2, neighbour table
constexpr uint32_t kOffA = 0, kOffB = 2 * kABytes, kOffP = kOffB + 2 * kBBytes, kOffU = kOffP + kRaw * kPBytes,
                   kOffY = kOffU + 2 * kUBytes, kSmemUsed = kOffY + 9 * kSites * 4;
constexpr size_t kSmem = kSmemUsed + 128;
constexpr int kOutStride = 51;                   // float2 per site of the transposed output (48 + 3: bank spread)
static_assert((kStageWarps + 1) * 12 * kOutStride * 8 <= kRaw * (int)kPBytes, "output staging");
static_assert(3 * kTileSites <= kRows && kTileSites <= kSites, "rows of a tile");
static_assert(kSmem <= 227 * 1024, "shared memory");

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t gtime() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ uint32_t core_off(int r, int k) {
    return (uint32_t)((r >> 3) * kSBO + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) |
           ((uint64_t)(kSBO >> 4) << 32) | ((uint64_t)1 << 46);
}
// D f32, A and B bf16, both K-major, N = 192, M = 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kN >> 3) << 17) |
                            ((uint32_t)(128 >> 4) << 24);

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait: true when the phase of the given parity has completed, false
// after wait_ns of global time (the context's wait limit) or 2^30 polls
__device__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned long long wait_ns) {
    const uint64_t t0 = gtime();
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        if (mbar_try(bar, parity)) return true;
        if ((it & 255u) == 255u && gtime() - t0 > wait_ns) return false;
    }
    return false;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {  // conj(a) b
    return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

// The raw rows of chunk j of warp `sg`'s sites into raw buffer j % kRaw, and with
// the first quarter of a transport its links into link buffer (transport & 1);
// one commit group per chunk (an empty one past the last).
__device__ __forceinline__ void gather(unsigned char* base, int sg, int lane, int j,
                                       const __nv_bfloat162* __restrict__ in, const float2* __restrict__ U32,
                                       int64_t xs0, int nsite) {
    if (j < kChunks) {
        const int d = j >> 2, qt = j & 3;
        const int* Y = (const int*)(base + kOffY) + d * kSites;
        const uint32_t P = su32(base + kOffP + (j % kRaw) * kPBytes);
#pragma unroll
        for (int t = 0; t < (kPieces + 31) / 32; ++t) {
            const int i = lane + 32 * t;
            const int sl = 8 * sg + i / 18, pc = i % 18;
            if (i < kPieces && sl < nsite)
                cp_async16(P + sl * kPStride + pc * 16,
                           (const unsigned char*)(in + ((int64_t)Y[sl] * kRC + kQ * qt) * 3) + pc * 16);
        }
        if (d > 0 && qt == 0) {
            const int mu = (d - 1) & 3;
            const uint32_t Ub = su32(base + kOffU + (d & 1) * kUBytes);
            for (int i = lane; i < 72; i += 32) {
                const int sl = 8 * sg + i / 9, e = i % 9;
                if (sl < nsite) {
                    const int64_t ls = d <= 4 ? xs0 + sl : (int64_t)Y[sl];
                    cp_async8(Ub + (sl * 9 + e) * 8, U32 + (ls * 4 + mu) * 9 + e);
                }
            }
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// two floats for the packed multiply-add
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ void fma2(uint64_t& r, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(r) : "l"(a), "l"(b));
}

// A lane's transport matrix, U (forward hop) or U^dag (backward hop), every
// component in both halves of a register pair.
struct Link2 {
    uint64_t x[9], y[9], ny[9];
};
__device__ __forceinline__ void load_link2(Link2& m, const float2* u, bool dagger) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float2 v = u[dagger ? 3 * c + a : 3 * a + c];
            const float im = dagger ? -v.y : v.y;
            m.x[3 * a + c] = pack2(v.x, v.x);
            m.y[3 * a + c] = pack2(im, im);
            m.ny[3 * a + c] = pack2(-im, -im);
        }
}

// Transport one chunk (24 input rows) of a lane's site: rows kq, kq + 4, ...;
// lane = (site j, kq).  A's rows are 3 site + colour; the bf16x2 stores of a warp
// land in 32 distinct banks (bank = 4 (row mod 8) + kq).
__device__ __forceinline__ uint32_t core_row(int r) { return (uint32_t)((r >> 3) * kSBO + (r & 7) * 16); }

__device__ __forceinline__ void stage_copy(const uint32_t* raw, unsigned char* a_s, int r0, int kq) {
#pragma unroll
    for (int h = 0; h < 6; ++h) {
        const uint32_t ok = (uint32_t)(h * 128 + 4 * kq);
#pragma unroll
        for (int c = 0; c < 3; ++c) *(uint32_t*)(a_s + core_row(r0 + c) + ok) = raw[(4 * h + kq) * 3 + c];
    }
}

__device__ __forceinline__ void stage_transport(const uint32_t* raw, const Link2& m, unsigned char* a_s, int r0,
                                                int kq) {
#pragma unroll
    for (int g = 0; g < 3; ++g) {
        uint64_t px[3], py[3];     // rows 8 g + kq and 8 g + 4 + kq
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const uint32_t w0 = raw[(8 * g + kq) * 3 + c], w1 = raw[(8 * g + 4 + kq) * 3 + c];
            px[c] = pack2(__uint_as_float(w0 << 16), __uint_as_float(w1 << 16));
            py[c] = pack2(__uint_as_float(w0 & 0xffff0000u), __uint_as_float(w1 & 0xffff0000u));
        }
        const uint32_t ok = (uint32_t)(2 * g * 128 + 4 * kq);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            uint64_t re = mul2(m.x[3 * a], px[0]), im = mul2(m.x[3 * a], py[0]);
            fma2(re, m.ny[3 * a], py[0]);
            fma2(im, m.y[3 * a], px[0]);
#pragma unroll
            for (int c = 1; c < 3; ++c) {
                fma2(re, m.x[3 * a + c], px[c]);
                fma2(im, m.x[3 * a + c], py[c]);
                fma2(re, m.ny[3 * a + c], py[c]);
                fma2(im, m.y[3 * a + c], px[c]);
            }
            const float2 r = unpack2(re), i = unpack2(im);
            *(__nv_bfloat162*)(a_s + core_row(r0 + a) + ok) = __floats2bfloat162_rn(r.x, i.x);
            *(__nv_bfloat162*)(a_s + core_row(r0 + a) + ok + 128) = __floats2bfloat162_rn(r.y, i.y);
        }
    }
}

__global__ void __launch_bounds__(kThreads, 1)
    k_net_conv_tc(const __nv_bfloat162* __restrict__ in, float2* __restrict__ out,
                  const __nv_bfloat16* __restrict__ Bw, const float2* __restrict__ U32,
                  const int2* __restrict__ nbr, int64_t V, int* err, unsigned long long wait_ns) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    // afull: the transport warps filled A stage s; bfull: B_j landed in B stage
    // s; mdone: the MMAs of the stage's chunk completed (tcgen05.commit)
    __shared__ __align__(8) uint64_t afull[2], bfull[2], mdone[2];
    __shared__ uint32_t tslot;
    __shared__ uint32_t committed;   // chunks whose MMAs warp 11 has committed
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&afull[s])), "r"(kStageWarps));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bfull[s])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&mdone[s])));
        }
        committed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(su32(&tslot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tslot;

    const int64_t ntiles = (V + kTileSites - 1) / kTileSites;
    uint32_t g = 0;  // chunks of the tiles before this one (stage = g & 1, use = g >> 1)
    int bad = 0;
    const int kq = lane & 3, sj = lane >> 2;
    for (int64_t tile = blockIdx.x; tile < ntiles && !bad; tile += gridDim.x) {
        const int64_t xs0 = tile * kTileSites;
        const int nsite = (int)(V - xs0 < kTileSites ? V - xs0 : kTileSites);
        // neighbour site of every (transport, site) of the tile
        int* Y = (int*)(base + kOffY);
        for (int i = tid; i < 9 * kSites; i += kThreads) {
            const int d = i / kSites, sl = i - d * kSites;
            if (sl < nsite) {
                const int64_t x = xs0 + sl;
                Y[i] = d == 0 ? (int)x : (d <= 4 ? __ldg(&nbr[x * 4 + d - 1].x) : __ldg(&nbr[x * 4 + d - 5].y));
            }
        }
        __syncthreads();
        if (warp < kStageWarps) {
            for (int j = 0; j < kRaw - 1; ++j) gather(base, warp, lane, j, in, U32, xs0, nsite);
            const int sl = 8 * warp + sj;
            Link2 m;
            for (int j = 0; j < kChunks; ++j) {
                const uint32_t gj = g + (uint32_t)j, s = gj & 1u, u = gj >> 1;
                // chunk j's raw rows are in, and the warp is done with chunk j - 1's,
                // whose buffer chunk j + 3 takes
                asm volatile("cp.async.wait_group %0;" ::"n"(kRaw - 2) : "memory");
                __syncwarp();
                gather(base, warp, lane, j + kRaw - 1, in, U32, xs0, nsite);
                // the MMAs of chunk gj - 2 read this A stage
                if (gj >= 2 && !mbar_wait(su32(&mdone[s]), (u - 1) & 1u, wait_ns)) bad = 1;
                if (__any_sync(0xffffffffu, bad)) {
                    bad = 1;
                    break;
                }
                const int d = j >> 2;
                const uint32_t* raw = (const uint32_t*)(base + kOffP + (j % kRaw) * kPBytes + sl * kPStride);
                unsigned char* a_s = base + kOffA + s * kABytes;
                if (sl < nsite) {
                    if (d == 0) {
                        stage_copy(raw, a_s, 3 * sl, kq);
                    } else {
                        if ((j & 3) == 0)
                            load_link2(m, (const float2*)(base + kOffU + (d & 1) * kUBytes) + sl * 9, d > 4);
                        stage_transport(raw, m, a_s, 3 * sl, kq);
                    }
                }
                // the tensor core reads the stage through the async proxy
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(&afull[s])) : "memory");
            }
        } else if (lane == 0) {
            // warp 11: B_j by bulk copy, then the chunk's MMAs once A and B are in
            for (int j = 0; j < kChunks; ++j) {
                const uint32_t gj = g + (uint32_t)j, s = gj & 1u, u = gj >> 1;
                if (gj >= 2 && !mbar_wait(su32(&mdone[s]), (u - 1) & 1u, wait_ns)) {  // B stage s free
                    bad = 1;
                    break;
                }
                const uint32_t bar = su32(&bfull[s]);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kBBytes)
                             : "memory");
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                        su32(base + kOffB + s * kBBytes)),
                    "l"(Bw + (size_t)j * (kBBytes / 2)), "r"(kBBytes), "r"(bar)
                    : "memory");
                if (!mbar_wait(su32(&afull[s]), u & 1u, wait_ns) || !mbar_wait(bar, u & 1u, wait_ns)) {
                    bad = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t a0 = su32(base + kOffA + s * kABytes), b0 = su32(base + kOffB + s * kBBytes);
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int ks = 0; ks < kKC / 16; ++ks) {
                        const uint64_t ad = sdesc(a0 + q * 16 * kSBO + ks * 256);
                        const uint64_t bd = sdesc(b0 + ks * 256);
                        const uint32_t acc = (j > 0 || ks > 0) ? 1u : 0u;
                        asm volatile(
                            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
                                tmem + (uint32_t)(q * kN)),
                            "l"(ad), "l"(bd), "r"(kIdesc), "r"(acc)
                            : "memory");
                    }
                asm volatile(
                    "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                        su32(&mdone[s]))
                    : "memory");
                committed = gj + 1;
            }
        }
        __syncwarp();
        // epilogue: the last chunk's commit covers every MMA of the tile
        if (tid == 0 && !bad) {
            const uint32_t gl = g + kChunks - 1;
            if (!mbar_wait(su32(&mdone[gl & 1u]), (gl >> 1) & 1u, wait_ns)) bad = 1;
        }
        g += kChunks;
        if (__syncthreads_or(bad)) bad = 1;
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (!bad) {
            // warp w reads lanes 32 (w % 4) .. + 31; the 12 (accumulator, 32 columns)
            // pieces of those lanes go to its three warps
            const int wq = warp & 3;
            float2* ot = (float2*)(base + kOffP) + warp * 12 * kOutStride;
            for (int u = warp >> 2; u < 2 * kN / 32; u += 3) {
                const int q = u / (kN / 32), c = 32 * (u - q * (kN / 32));
                const int r = 128 * q + 32 * wq + lane;
                uint32_t v[32];
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                    "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                      "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
                      "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
                      "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
                      "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                    : "r"(tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)(q * kN + c)));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                // a site's 16 x 3 numbers are contiguous in memory: transposed through
                // shared memory (the raw buffers are done with), a store covers whole lines
                const int f = r / 3, f0 = (128 * q + 32 * wq) / 3;
                float2* o = ot + (f - f0) * kOutStride + (r - 3 * f);
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    o[3 * i] = make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
                __syncwarp();
                float2* dst = out + ((xs0 + f0) * kRC + c / 2) * 3;
#pragma unroll 6
                for (int t = lane; t < 12 * 48; t += 32) {
                    const int fl = t / 48, w = t - fl * 48;
                    const int rr = 3 * (f0 + fl) + w % 3 - (r - lane);   // the row's lane
                    if (rr >= 0 && rr < 32 && f0 + fl < nsite) dst[fl * (3 * kRC) + w] = ot[fl * kOutStride + w];
                }
                __syncwarp();
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        if (__syncthreads_or(bad)) bad = 1;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (bad && tid == 0) atomicExch(err, 1);
    // every committed MMA has been waited for on the normal path; after a
    // timeout give the in-flight ones a bounded time before freeing
    __syncthreads();
    if (bad && tid == 0 && committed > 0) {
        const uint32_t gl = committed - 1;
        mbar_wait(su32(&mdone[gl & 1u]), (gl >> 1) & 1u, wait_ns);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// B chunks from the FP32 master weights WT[d][k][R] (complex, transposed)
__global__ void k_net_tc_pack(const float2* __restrict__ WT, __nv_bfloat16* __restrict__ Bw) {
    const int64_t n = (int64_t)kChunks * kN * kKC;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int chunk = (int)(e / (kN * kKC));
        const int rem = (int)(e - (int64_t)chunk * kN * kKC);
        const int np = rem / kKC, kp = rem - np * kKC;
        const int d = chunk >> 2, qt = chunk & 3;
        const int o = np >> 1, cout = np & 1, kk = kp >> 1, cin = kp & 1;
        const int k = kQ * qt + kk;
        const float2 w = WT[((int64_t)d * kRC + k) * kRC + o];
        const float v = cout == 0 ? (cin == 0 ? w.x : -w.y) : (cin == 0 ? w.y : w.x);
        Bw[(int64_t)chunk * (kBBytes / 2) + core_off(np, kp) / 2] = __float2bfloat16_rn(v);
    }
}

// ---------------------------------------------------------------------------
// The C -> 1 layer, weights first, on the tensor cores:
//   Phi[y][d][R][b] = sum_k W_d[R, k] in(y)[k, b]
// a real GEMM over rows p = 3 y + b with K = 2 x 96 (k' = 2 k + (re, im)) and
// N = 72 real outputs n' = 2 (4 d + R) + (re, im), padded to 80.  No
// transport: the A rows are the site's own activations (FP32, contiguous),
// converted to BF16 into the core-matrix layout.  128 rows per tile, one
// 80-column accumulator; 78 KB of shared memory and 128 TMEM columns, so two
// CTAs share an SM and overlap one's staging with the other's MMA/epilogue.
// ---------------------------------------------------------------------------
constexpr int kPhiRows = 128;
constexpr int kPhiK = 192;
constexpr int kPhiN = 80;
constexpr int kPhiOut = 72;
constexpr uint32_t kPhiSBO = (kPhiK / 8) * 128;          // 3072
constexpr uint32_t kPhiABytes = kPhiRows * kPhiK * 2;    // 49152
constexpr uint32_t kPhiBBytes = kPhiN * kPhiK * 2;       // 30720
constexpr size_t kPhiSmem = kPhiABytes + kPhiBBytes + 128;
constexpr int kPhiThreads = 256;
constexpr uint32_t kPhiIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kPhiN >> 3) << 17) |
                               ((uint32_t)(kPhiRows >> 4) << 24);

__device__ __forceinline__ uint32_t phi_off(int r, int k) {
    return (uint32_t)((r >> 3) * kPhiSBO + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}
__device__ __forceinline__ uint64_t phi_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) |
           ((uint64_t)(kPhiSBO >> 4) << 32) | ((uint64_t)1 << 46);
}

__global__ void __launch_bounds__(kPhiThreads, 2)
    k_net_phi_tc(const float2* __restrict__ in, float2* __restrict__ phi, const __nv_bfloat16* __restrict__ Bw,
                 int64_t V, int* err, unsigned long long wait_ns) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    unsigned char* sA = base;
    unsigned char* sB = base + kPhiABytes;
    __shared__ __align__(8) uint64_t bfull, mdone;
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bfull)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&mdone)));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(su32(&tslot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tslot;
    if (tid == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(&bfull)), "r"(kPhiBBytes)
                     : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         su32(sB)),
                     "l"(Bw), "r"(kPhiBBytes), "r"(su32(&bfull))
                     : "memory");
    }
    const int64_t rows = 3 * V;
    const int64_t ntiles = (rows + kPhiRows - 1) / kPhiRows;
    int bad = 0;
    uint32_t used = 0;  // tiles whose MMAs this CTA committed
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t row0 = tile * kPhiRows;
        const int64_t y0 = row0 / 3;
        int64_t yl = (row0 + kPhiRows - 1) / 3;
        if (yl > V - 1) yl = V - 1;
        const int nsite = (int)(yl - y0 + 1);
        const int off = (int)(row0 - 3 * y0);
        // A: the tile's sites' activations, contiguous in memory ([y][k][b])
        // thread = (site, k): the three colours are three rows of the tile
        for (int e = tid; e < nsite * kRC; e += kPhiThreads) {
            const int sl = e / kRC, k = e - sl * kRC;
            const float2* src = in + ((y0 + sl) * kRC + k) * 3;
            const float2 v0 = __ldg(src), v1 = __ldg(src + 1), v2 = __ldg(src + 2);
            const int r = 3 * sl - off;
            if (r >= 0 && r < kPhiRows)
                *(__nv_bfloat162*)(sA + phi_off(r, 2 * k)) = __floats2bfloat162_rn(v0.x, v0.y);
            if (r + 1 >= 0 && r + 1 < kPhiRows)
                *(__nv_bfloat162*)(sA + phi_off(r + 1, 2 * k)) = __floats2bfloat162_rn(v1.x, v1.y);
            if (r + 2 < kPhiRows)
                *(__nv_bfloat162*)(sA + phi_off(r + 2, 2 * k)) = __floats2bfloat162_rn(v2.x, v2.y);
        }
        // rows past the last site (the last tile only) are zero
        for (int e = tid; e < kPhiRows * kRC; e += kPhiThreads) {
            const int r = e / kRC, k = e - r * kRC;
            if (row0 + r >= rows)
                *(__nv_bfloat162*)(sA + phi_off(r, 2 * k)) = __floats2bfloat162_rn(0.f, 0.f);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            if ((used == 0 && !mbar_wait(su32(&bfull), 0u, wait_ns))) {
                bad = 1;
            } else {
                asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
                for (int ks = 0; ks < kPhiK / 16; ++ks) {
                    const uint64_t ad = phi_desc(su32(sA) + ks * 256);
                    const uint64_t bd = phi_desc(su32(sB) + ks * 256);
                    const uint32_t acc = ks > 0 ? 1u : 0u;
                    asm volatile(
                        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
                        "l"(ad), "l"(bd), "r"(kPhiIdesc), "r"(acc)
                        : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 su32(&mdone))
                             : "memory");
            }
        }
        if (__syncthreads_or(bad)) {
            bad = 1;
            break;
        }
        ++used;
        if (!mbar_wait(su32(&mdone), (used - 1) & 1u, wait_ns)) bad = 1;
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (!__syncthreads_or(bad)) {
            // warp w: lanes 32 (w % 4) .. + 31, columns 40 (w / 4) .. + 39
            const int wq = warp & 3, ch = warp >> 2;
            const int r = 32 * wq + lane;
            const int64_t p = row0 + r;
            const int64_t y = p / 3;
            const int b = (int)(p - 3 * y);
#pragma unroll
            for (int c8 = 0; c8 < 5; ++c8) {
                const int c = 40 * ch + 8 * c8;
                uint32_t v[8];
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                             : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                               "=r"(v[6]), "=r"(v[7])
                             : "r"(tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)c));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (p < rows) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int dR = c / 2 + i;
                        if (dR < kPhiOut / 2)
                            phi[(y * (kPhiOut / 2) + dR) * 3 + b] =
                                make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
                    }
                }
            }
        } else {
            bad = 1;
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        if (__syncthreads_or(bad)) {
            bad = 1;
            break;
        }
    }
    if (bad && tid == 0) atomicExch(err, 1);
    // the weight copy must have landed before the CTA exits
    if (tid == 0 && used == 0) mbar_wait(su32(&bfull), 0u, wait_ns);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem));
}

// B of the C -> 1 layer from its FP32 master weights WT[d][k][R] (R < 4)
__global__ void k_net_phi_pack(const float2* __restrict__ WT, __nv_bfloat16* __restrict__ Bw) {
    const int n = kPhiN * kPhiK;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const int np = e / kPhiK, kp = e - np * kPhiK;
        float v = 0.f;
        if (np < kPhiOut) {
            const int o = np >> 1, cout = np & 1, k = kp >> 1, cin = kp & 1;
            const int d = o >> 2, R = o & 3;
            const float2 w = WT[((int64_t)d * kRC + k) * 4 + R];
            v = cout == 0 ? (cin == 0 ? w.x : -w.y) : (cin == 0 ? w.y : w.x);
        }
        Bw[phi_off(np, kp) / 2] = __float2bfloat16_rn(v);
    }
}

// ---------------------------------------------------------------------------
// The 1 -> C layer on the tensor cores: rows p = 3 x + a, K = 9 transports x
// 4 spins x (re, im) = 72 (padded to 80, the padding columns of A zero once),
// N = 192 (96 outputs x (re, im)); the threads stage U_d(x) in(x + d) for the
// 4 input rows (FP32 links and activations through L1); BF16 output in the
// layout the C -> C layer reads ([V][96][3] bf16x2).  128 rows per tile,
// weights resident (30 KB), 192 TMEM columns, two CTAs per SM.
// ---------------------------------------------------------------------------
constexpr int kL1Rows = 128;
constexpr int kL1K = 80;
constexpr uint32_t kL1SBO = (kL1K / 8) * 128;          // 1280
constexpr uint32_t kL1ABytes = kL1Rows * kL1K * 2;     // 20480
constexpr uint32_t kL1BBytes = kN * kL1K * 2;          // 30720
constexpr size_t kL1Smem = kL1ABytes + kL1BBytes + 128;
constexpr int kL1Threads = 256;
constexpr uint32_t kL1Idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kN >> 3) << 17) |
                              ((uint32_t)(kL1Rows >> 4) << 24);

__device__ __forceinline__ uint32_t l1_off(int r, int k) {
    return (uint32_t)((r >> 3) * kL1SBO + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}
__device__ __forceinline__ uint64_t l1_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) |
           ((uint64_t)(kL1SBO >> 4) << 32) | ((uint64_t)1 << 46);
}

__global__ void __launch_bounds__(kL1Threads, 2)
    k_net_l1_tc(const float2* __restrict__ in, __nv_bfloat162* __restrict__ out, const __nv_bfloat16* __restrict__ Bw,
                const float2* __restrict__ U32, const int2* __restrict__ nbr, int64_t V, int* err,
                unsigned long long wait_ns) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    unsigned char* sA = base;
    unsigned char* sB = base + kL1ABytes;
    __shared__ __align__(8) uint64_t bfull, mdone;
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bfull)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&mdone)));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(su32(&tslot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // the padding columns 72..79 of A stay zero
    for (int r = tid; r < kL1Rows; r += kL1Threads) {
        *(uint4*)(sA + l1_off(r, 72)) = make_uint4(0u, 0u, 0u, 0u);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tslot;
    if (tid == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(&bfull)), "r"(kL1BBytes)
                     : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         su32(sB)),
                     "l"(Bw), "r"(kL1BBytes), "r"(su32(&bfull))
                     : "memory");
    }
    const int64_t rows = 3 * V;
    const int64_t ntiles = (rows + kL1Rows - 1) / kL1Rows;
    int bad = 0;
    uint32_t used = 0;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t row0 = tile * kL1Rows;
        const int64_t x0 = row0 / 3;
        int64_t xl = (row0 + kL1Rows - 1) / 3;
        if (xl > V - 1) xl = V - 1;
        const int nsite = (int)(xl - x0 + 1);
        const int off = (int)(row0 - 3 * x0);
        // A: item = (site, transport): 4 input rows x 3 colours
        for (int e = tid; e < nsite * 9; e += kL1Threads) {
            const int sl = e / 9, d = e - sl * 9;
            const int64_t x = x0 + sl;
            int64_t y = x;
            const float2* uu = nullptr;
            bool dag = false;
            if (d >= 1 && d <= 4) {
                y = __ldg(&nbr[x * 4 + d - 1].x);
                uu = U32 + (x * 4 + d - 1) * 9;
            } else if (d >= 5) {
                y = __ldg(&nbr[x * 4 + d - 5].y);
                uu = U32 + (y * 4 + d - 5) * 9;
                dag = true;
            }
            float2 u[9];
            if (uu) {
#pragma unroll
                for (int i = 0; i < 9; ++i) u[i] = __ldg(uu + i);
            }
            const float2* src = in + y * 12;
            const int r0 = 3 * sl - off;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 p0 = __ldg(src + 3 * k), p1 = __ldg(src + 3 * k + 1), p2 = __ldg(src + 3 * k + 2);
                float2 t[3];
                if (!uu) {
                    t[0] = p0;
                    t[1] = p1;
                    t[2] = p2;
                } else if (!dag) {
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const float2 q0 = cmul(u[3 * a], p0), q1 = cmul(u[3 * a + 1], p1), q2 = cmul(u[3 * a + 2], p2);
                        t[a] = make_float2(q0.x + q1.x + q2.x, q0.y + q1.y + q2.y);
                    }
                } else {
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const float2 q0 = cmulc(u[a], p0), q1 = cmulc(u[3 + a], p1), q2 = cmulc(u[6 + a], p2);
                        t[a] = make_float2(q0.x + q1.x + q2.x, q0.y + q1.y + q2.y);
                    }
                }
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int r = r0 + a;
                    if (r >= 0 && r < kL1Rows)
                        *(__nv_bfloat162*)(sA + l1_off(r, 2 * (4 * d + k))) = __floats2bfloat162_rn(t[a].x, t[a].y);
                }
            }
        }
        // rows past the last site (the last tile only) are zero
        for (int e = tid; e < kL1Rows * 36; e += kL1Threads) {
            const int r = e / 36, q = e - r * 36;
            if (row0 + r >= rows) *(__nv_bfloat162*)(sA + l1_off(r, 2 * q)) = __floats2bfloat162_rn(0.f, 0.f);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            if (used == 0 && !mbar_wait(su32(&bfull), 0u, wait_ns)) {
                bad = 1;
            } else {
                asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
                for (int ks = 0; ks < kL1K / 16; ++ks) {
                    const uint64_t ad = l1_desc(su32(sA) + ks * 256);
                    const uint64_t bd = l1_desc(su32(sB) + ks * 256);
                    const uint32_t acc = ks > 0 ? 1u : 0u;
                    asm volatile(
                        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
                        "l"(ad), "l"(bd), "r"(kL1Idesc), "r"(acc)
                        : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 su32(&mdone))
                             : "memory");
            }
        }
        if (__syncthreads_or(bad)) {
            bad = 1;
            break;
        }
        ++used;
        if (!mbar_wait(su32(&mdone), (used - 1) & 1u, wait_ns)) bad = 1;
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (!__syncthreads_or(bad)) {
            // warp w: lanes 32 (w % 4) .. + 31, columns 96 (w / 4) .. + 95
            const int wq = warp & 3, ch = warp >> 2;
            const int r = 32 * wq + lane;
            const int64_t p = row0 + r;
            const int64_t x = p / 3;
            const int a = (int)(p - 3 * x);
            for (int c = 96 * ch; c < 96 * ch + 96; c += 32) {
                uint32_t v[32];
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                    "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                      "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
                      "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
                      "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
                      "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                    : "r"(tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)c));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (p < rows) {
                    __nv_bfloat162* dst = out + (x * kRC + c / 2) * 3 + a;
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        dst[3 * i] = __floats2bfloat162_rn(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
                }
            }
        } else {
            bad = 1;
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        if (__syncthreads_or(bad)) {
            bad = 1;
            break;
        }
    }
    if (bad && tid == 0) atomicExch(err, 1);
    if (tid == 0 && used == 0) mbar_wait(su32(&bfull), 0u, wait_ns);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem));
}

// B of the 1 -> C layer from its FP32 master weights WT[d][k][R] (k < 4)
__global__ void k_net_l1_pack(const float2* __restrict__ WT, __nv_bfloat16* __restrict__ Bw) {
    const int n = kN * kL1K;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const int np = e / kL1K, kp = e - np * kL1K;
        float v = 0.f;
        if (kp < 72) {
            const int o = np >> 1, cout = np & 1, q = kp >> 1, cin = kp & 1;
            const int d = q >> 2, k = q & 3;
            const float2 w = WT[((int64_t)d * 4 + k) * kRC + o];
            v = cout == 0 ? (cin == 0 ? w.x : -w.y) : (cin == 0 ? w.y : w.x);
        }
        Bw[l1_off(np, kp) / 2] = __float2bfloat16_rn(v);
    }
}

// Failure-detection self-test: one thread waits, through the same bounded
// mbar_wait as the kernels above, on an mbarrier that nothing ever arrives
// at; the wait runs out after wait_ns and the kernel records GS_TIMEOUT.
__global__ void k_selftest_mbar_timeout(int* err, unsigned long long wait_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&bar)));
        asm volatile("fence.mbarrier_init.release.cluster;");
        if (!mbar_wait(su32(&bar), 0u, wait_ns)) atomicExch(err, (int)GS_TIMEOUT);
        asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(su32(&bar)));
    }
}

}  // namespace

size_t net_tc_weight_elems() { return (size_t)kChunks * kN * kKC; }

gs_status net_tc_pack(gs_ctx* c, const float2* WT, __nv_bfloat16* Bw) {
    k_net_tc_pack<<<grid_for((int64_t)net_tc_weight_elems(), 256, c->num_sms * 4), 256, 0, c->stream>>>(WT, Bw);
    c->launches++;
    GS_CHECK_LAUNCH(c);
    return GS_OK;
}

size_t net_phi_weight_elems() { return (size_t)kPhiN * kPhiK; }
size_t net_l1_weight_elems() { return (size_t)kN * kL1K; }

gs_status net_l1_pack(gs_ctx* c, const float2* WT, __nv_bfloat16* Bw) {
    k_net_l1_pack<<<grid_for(kN * kL1K, 256, 64), 256, 0, c->stream>>>(WT, Bw);
    c->launches++;
    GS_CHECK_LAUNCH(c);
    return GS_OK;
}

gs_status net_l1_tc(gs_ctx* c, const float2* in, __nv_bfloat162* out, const __nv_bfloat16* Bw, const float2* U32,
                    const int2* nbr, int64_t V, int* err) {
    GS_CUDA(c, cudaFuncSetAttribute(k_net_l1_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kL1Smem));
    const int64_t ntiles = (3 * V + kL1Rows - 1) / kL1Rows;
    const int64_t cap = 2LL * c->num_sms;
    const int grid = (int)(ntiles < cap ? ntiles : cap);
    k_net_l1_tc<<<grid, kL1Threads, kL1Smem, c->stream>>>(in, out, Bw, U32, nbr, V, err, c->wait_ns);
    c->launches++;
    GS_CHECK_LAUNCH(c);
    return GS_OK;
}

gs_status net_phi_pack(gs_ctx* c, const float2* WT, __nv_bfloat16* Bw) {
    k_net_phi_pack<<<grid_for(kPhiN * kPhiK, 256, 64), 256, 0, c->stream>>>(WT, Bw);
    c->launches++;
    GS_CHECK_LAUNCH(c);
    return GS_OK;
}

gs_status net_phi_tc(gs_ctx* c, const float2* in, float2* phi, const __nv_bfloat16* Bw, int64_t V, int* err) {
    GS_CUDA(c, cudaFuncSetAttribute(k_net_phi_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPhiSmem));
    const int64_t ntiles = (3 * V + kPhiRows - 1) / kPhiRows;
    const int64_t cap = 2LL * c->num_sms;
    const int grid = (int)(ntiles < cap ? ntiles : cap);
    k_net_phi_tc<<<grid, kPhiThreads, kPhiSmem, c->stream>>>(in, phi, Bw, V, err, c->wait_ns);
    c->launches++;
    GS_CHECK_LAUNCH(c);
    return GS_OK;
}

gs_status net_conv_tc(gs_ctx* c, const __nv_bfloat162* in, float2* out, const __nv_bfloat16* Bw, const float2* U32,
                      const int2* nbr, int64_t V, int* err) {
    GS_CUDA(c, cudaFuncSetAttribute(k_net_conv_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
    const int64_t ntiles = (V + kTileSites - 1) / kTileSites;
    const int grid = (int)(ntiles < c->num_sms ? ntiles : c->num_sms);
    k_net_conv_tc<<<grid, kThreads, kSmem, c->stream>>>(in, out, Bw, U32, nbr, V, err, c->wait_ns);
    c->launches++;
    GS_CHECK_LAUNCH(c);
    return GS_OK;
}

// Runs k_selftest_mbar_timeout; *err_dev receives GS_TIMEOUT when the wait ran out.
gs_status selftest_mbar_timeout(gs_ctx* c, int* err_dev) {
    k_selftest_mbar_timeout<<<1, 32, 0, c->stream>>>(err_dev, c->wait_ns);
    c->launches++;
    GS_CHECK_LAUNCH(c);
    return GS_OK;
}

}  // namespace gs
