// FP64 Wilson-Dirac stencil on label-ordered vectors, restricted to label
// ranges: the blocks D_bb, D_br, D_rb, D_rr of the permuted operator P D P^T
// (Section 1 of the paper: the 2x2 partition) and the full D (identity plan).
//
//   (D psi)(x) = (m0 + 4) psi(x) - 1/2 sum_mu [ (1 - g_mu) U_mu(x) psi(x+mu)
//                                   + (1 + g_mu) U_mu(x-mu)^dag psi(x-mu) ]
//
// gamma matrices in the DeGrand-Rossi chiral basis: g_mu = [[0, X], [X^dag, 0]]
// with X_0 = [[0,i],[i,0]], X_1 = [[0,-1],[1,0]], X_2 = diag(i,-i), X_3 = 1.
// Then (1 -+ g_mu) psi = [h; -+ X^dag h] with h = psi_up -+ X psi_lo, so each hop
// multiplies only the two-spinor h by the link (spin projection) and the
// lower half of the result is X^dag applied to (g_back - g_fwd).
//
// FP64 runs at ~1/60 of the FP32 rate on this part.  A context's stencils
// therefore do the same operator in integer arithmetic (dslash_fx.cu: 8^4 8.2 us
// against 12.3, 24^3 x 48 0.50 ms against 1.03); the double-precision kernel here
// serves the entry point that allocates nothing and fields whose links fixed
// point cannot hold, and its tile (dslash_f64.cuh) vectors that it cannot hold (in the
// fixed-point kernel only 4 of a block's 8 or 16 warps work on that tile: a whole
// field of them took 14.4 us on 8^4 and 1.20 ms on 24^3 x 48, here 12.3 us and 1.03 ms).
// It is bound by the FP64 pipe: a
// block of 4 warps covers 32 sites and warp w handles direction mu = w (forward
// and backward hop) for all 32 sites, so the spin projection specialises without
// divergence; the four partial 24-double results meet in shared memory (SoA,
// bank-conflict free) and warp w then finishes spin component w of the 32 sites.
// Links are stored pre-multiplied by -1/2 (exact in binary).
#include "dslash_f64.cuh"

namespace gs {

namespace {

template <int EPI>
__global__ void __launch_bounds__(kThreads) k_dslash_f64(StencilArgs a) {
    const bool skip = a.st != nullptr && a.st->done;
    if (a.ran != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *a.ran = skip ? 0 : 1;
    if (skip) return;
    __shared__ double red[4][24][kSitesPerBlock];
    double e[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int64_t base = (int64_t)blockIdx.x * kSitesPerBlock; base < a.n_out;
         base += (int64_t)gridDim.x * kSitesPerBlock)
        f64_tile<EPI>(a, base, kSitesPerBlock, red, e);
    stencil_finish<EPI, kThreads>(a, e);
}

}  // namespace

gs_status launch_stencil_f64(gs_ctx* c, const StencilArgs& args) {
    if (args.n_out <= 0) return GS_OK;
    StencilArgs a = args;
    int slot = -1;
    if (c->prof.on) {
        gs_status s = prof_begin(c, &slot);
        if (s != GS_OK) return s;
        a.ran = c->prof.ran_dev + slot;
    } else {
        a.ran = nullptr;
    }
    const int64_t blocks_needed = (a.n_out + kSitesPerBlock - 1) / kSitesPerBlock;
    int max_blocks = (a.epi == EPI_NONE) ? (1 << 30) : kMaxRedBlocks;
    const int g = (int)(blocks_needed < max_blocks ? blocks_needed : max_blocks);
    if (!c->fx_m || plan_fits(a.plan) == 0) {
        switch (a.epi) {
            case EPI_NONE: k_dslash_f64<EPI_NONE><<<g, kThreads, 0, c->stream>>>(a); break;
            case EPI_DOT_RHAT_V: k_dslash_f64<EPI_DOT_RHAT_V><<<g, kThreads, 0, c->stream>>>(a); break;
            default: k_dslash_f64<EPI_DOT_TS><<<g, kThreads, 0, c->stream>>>(a); break;
        }
        c->launches++;
    } else {   // where the host does not know yet, the kernel looks at the flag itself
        fx_args(a.plan, c->fx_m, c->fx_e, a.b1 - a.a0, &a);
        gs_status s = launch_stencil_fx(c, a, g);
        if (s != GS_OK) return s;
    }
    c->stencil_sites += a.n_out;
    GS_CHECK_LAUNCH(c);
    if (slot >= 0) return prof_end(c, slot, a.plan, a);
    return GS_OK;
}

// The double-precision kernel on a caller's stream without a context: used by
// the entry point that allocates nothing, which has no room for a fixed-point
// copy of the links and the input.
gs_status launch_stencil_f64_on(const StencilArgs& args, cudaStream_t stream) {
    if (args.n_out <= 0) return GS_OK;
    StencilArgs a = args;
    a.ran = nullptr;
    a.epi = EPI_NONE;
    a.st = nullptr;
    const int64_t g = (a.n_out + kSitesPerBlock - 1) / kSitesPerBlock;
    k_dslash_f64<EPI_NONE><<<(int)g, kThreads, 0, stream>>>(a);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ECUDA;
}

}  // namespace gs
