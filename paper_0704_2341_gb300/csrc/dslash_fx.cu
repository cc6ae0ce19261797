// The FP64 Wilson stencil in block fixed point (fx.cuh, dslash_fx.cuh): a
// kernel that turns the input vector into fixed point and the stencil itself.
#include "dslash_fx.cuh"

namespace gs {
namespace {

// Fixed-point copy of the stencil input of n sites (the first nA at A, the
// rest at B, complex128 [site][12]): mantissas in groups of 32 sites (fx_index),
// so that the stencil's neighbour loads are whole lines, and one exponent per site.
// The two kernels of a stencil call are launched back to back; the second one
// starts early and waits for this one's results (programmatic launch).
__global__ void __launch_bounds__(kThreads) k_fx_pack(const double2* __restrict__ A, int64_t nA,
                                                      const double2* __restrict__ B, int64_t n,
                                                      longlong2* __restrict__ m, int* __restrict__ ex) {
    asm volatile("griddepcontrol.launch_dependents;");
    __shared__ double2 sm[32][13];
    __shared__ int smax[4][32], sden[4][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int64_t base = (int64_t)blockIdx.x * 32; base < n; base += (int64_t)gridDim.x * 32) {
        const int64_t left = n - base;
        const int cnt = (int)(left < 32 ? left : 32) * kSiteC;
        for (int i = threadIdx.x; i < cnt; i += kThreads) {
            const int site = i / kSiteC;
            const double2* src = base + site < nA ? A + base * kSiteC : B + (base - nA) * kSiteC;
            sm[site][i - site * kSiteC] = __ldg(src + i);
        }
        __syncthreads();
        unsigned hi[6], lo[6];
        int e = 0;
        unsigned any = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 v = sm[lane][3 * warp + c];
            hi[2 * c] = (unsigned)__double2hiint(v.x);
            lo[2 * c] = (unsigned)__double2loint(v.x);
            hi[2 * c + 1] = (unsigned)__double2hiint(v.y);
            lo[2 * c + 1] = (unsigned)__double2loint(v.y);
            e = max(e, max(fx_exponent(hi[2 * c]), fx_exponent(hi[2 * c + 1])));
            any |= ((hi[2 * c] | hi[2 * c + 1]) & 0x7fffffffu) | lo[2 * c] | lo[2 * c + 1];
        }
        smax[warp][lane] = e;
        sden[warp][lane] = any != 0;
        __syncthreads();
        const int E = max(max(smax[0][lane], smax[1][lane]), max(smax[2][lane], smax[3][lane]));
        const bool zero = !(sden[0][lane] | sden[1][lane] | sden[2][lane] | sden[3][lane]);
        if (base + lane < n) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
                m[base * kSiteC + (3 * warp + c) * 32 + lane] =
                    make_longlong2(fx_from_bits(hi[2 * c], lo[2 * c], E), fx_from_bits(hi[2 * c + 1], lo[2 * c + 1], E));
            if (warp == 0) ex[base + lane] = zero ? kFxZero : (E < kFxMinExp || E > kFxMaxExp) ? kFxBad : E;
        }
        __syncthreads();
    }
}

template <int EPI, int NS, bool KEEP>
__global__ void __launch_bounds__(kFxThreads<NS>, NS) k_dslash_fx(const __grid_constant__ StencilArgs a) {
    __shared__ FxShared sm;
    __shared__ int sE[8][kSitesPerBlock];
    __shared__ unsigned redo[KEEP ? kFxRedoWords : 1];
    const int l = fx_label(a, (int64_t)blockIdx.x * kSitesPerBlock, kSitesPerBlock, (threadIdx.x >> 5) * NS);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const bool skip = a.st != nullptr && a.st->done;
    if (a.ran != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *a.ran = skip ? 0 : 1;
    if (skip) return;
    const bool links_bad = __ldg(a.fxflag) != 0;
    double e[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    fx_stencil<EPI, NS, KEEP>(a, links_bad, sm, sE, redo, l, e);
    stencil_finish<EPI, kFxThreads<NS>>(a, e);
}

// Up to two tiles an SM a short call wants the shortest tile (8^4: 8.2 us with 16
// warps a tile against 10.2 with 8); beyond that the integer pipes are the
// bound and 8 warps a tile issue fewer instructions a site (24^3 x 48: 0.50 ms
// against 0.61).
template <int NS>
cudaError_t launch_fx(const StencilArgs& a, cudaLaunchConfig_t cfg, int grid, int sms) {
    const int64_t tiles = (a.n_out + kSitesPerBlock - 1) / kSitesPerBlock;
    const int least = (int)((tiles + 32 * kFxRedoWords - 1) / (32 * kFxRedoWords));   // blocks whose tiles fit `redo`
    const int most = NS * sms > least ? NS * sms : least;
    cfg.gridDim = dim3(grid < most ? grid : most);
    cfg.blockDim = dim3(kFxThreads<NS>);
    switch (a.epi) {
        case EPI_NONE:
            return cudaLaunchKernelEx(&cfg, a.keep_weak ? k_dslash_fx<EPI_NONE, NS, true> : k_dslash_fx<EPI_NONE, NS, false>, a);
        case EPI_DOT_RHAT_V: return cudaLaunchKernelEx(&cfg, k_dslash_fx<EPI_DOT_RHAT_V, NS, false>, a);
        default: return cudaLaunchKernelEx(&cfg, k_dslash_fx<EPI_DOT_TS, NS, false>, a);
    }
}

}  // namespace

void fx_args(const Plan* p, const longlong2* m, const int* e, int64_t n, StencilArgs* a) {
    a->fxm = m;
    a->fxe = e;
    a->fxn = n;
    a->fxl = p->fx_links;
    a->fxflag = p->fx_flag;
}

gs_status launch_stencil_fx(gs_ctx* c, const StencilArgs& a, int grid) {
    const int64_t n = a.fxn;
    const int gp = grid_for(n, 32, 1 << 30);
    k_fx_pack<<<gp, kThreads, 0, c->stream>>>(a.inA, a.a1 - a.a0, a.inB, n, c->fx_m, c->fx_e);
    GS_CHECK_LAUNCH(c);
    cudaLaunchConfig_t cfg = {};
    cfg.stream = c->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = grid <= 2 * c->num_sms ? launch_fx<1>(a, cfg, grid, c->num_sms)
                                                 : launch_fx<2>(a, cfg, grid, c->num_sms);
    if (e != cudaSuccess) return set_err(c, GS_ECUDA, "stencil launch failed: %s", cudaGetErrorString(e));
    c->launches += 2;
    return GS_OK;
}

}  // namespace gs
