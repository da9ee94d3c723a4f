// Transport kernels (sm_103a) of the state, adjoint, incremental state and incremental adjoint
// equations of Mang & Biros (arXiv 1503.00757, Sec. 3) on a 2-D grid: Heun's RK2 in pseudo-time
// with spectral derivatives taken axis by axis (deriv.cuh).
//
// Bound by the latency of a chain of dependent launches (64 to 128 CTAs of a few microseconds at
// 512^2), so what counts is what lies between one launch's wait and its last store: the row
// kernels' transforms precede their wait, no spectra are split or merged, and the operands are in
// registers when the column kernel's result arrives.  512^2, nt = 32 matvec: 1464 us with the
// stages in the row spectra, 848 us with these (6.3 us a stage).
#include <type_traits>

#include "deriv.cuh"
#include "internal.h"
#include "launch.cuh"

// ---------------------------------------------------------------------------
// transport kernels: one RK2 (Heun) stage is a column kernel (the x^1 derivative of the stage's
// field, deriv.cuh) and a row kernel (the x^2 derivative and the update).  Fields travel as plain
// real fields: the derivative along an axis needs no transform of the other one.
// ---------------------------------------------------------------------------
// blockIdx.y: independent fields, bs floats apart
template <int LOGL, int LC>
__global__ void __launch_bounds__(256) k_dcol(DColArgs a, ColMap m, long long bs, const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    a.f += blockIdx.y * bs;
    a.out += blockIdx.y * bs;
    dcol_body<LOGL, LC, true>(a, m, blockIdx.x, sm, tw, pdl_entry);
}

// PRE (deriv.cuh): needs about 130 registers a thread; without it the kernel is held to 64, which
// many concurrent solves may want: the autotuner chooses per grid.  Rows of 1024 points have the
// PRE variant only (64 x 1024, nt = 16 matvec: 578 us without).
template <int LOGL, bool PRE>
__global__ void __launch_bounds__(256, PRE ? 1 : 4) k_adv_row(AdvStage<2> a, int N, int lines,
                                                              const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    adv_row_body<LOGL, 2, PRE, 2>(a, (uint32_t)N, lines, sm, tw, pdl_entry);
}

template <int LOGL, bool PRE, bool FULL>
__global__ void __launch_bounds__(256, PRE ? 1 : (FULL ? 3 : 4)) k_adj_row(AdjStage<2> a, int N, int lines,
                                                                          const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    adj_row_body<LOGL, 2, PRE, FULL, 2>(a, (uint32_t)N, lines, sm, tw, pdl_entry);
}

// lam(1) = ca a + cb c (a nullable) and b = w lam grad m(1); with lsrc (full Newton) b += w lsrc gmt
__global__ void __launch_bounds__(NTHREADS) k_adj_init(const float* __restrict__ a, float ca,
                                                       const float* __restrict__ c, float cb, float* lam, float* b,
                                                       const float* __restrict__ gm, float w,
                                                       const float* __restrict__ lsrc, const float* __restrict__ gmt,
                                                       int N) {
    pdl_entry();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        float l = cb * c[i];
        if (a) l = fmaf(ca, a[i], l);
        lam[i] = l;
        float b1 = w * l * gm[i], b2 = w * l * gm[N + i];
        if (lsrc) {
            const float ls = w * lsrc[i];
            b1 = fmaf(ls, gmt[i], b1);
            b2 = fmaf(ls, gmt[N + i], b2);
        }
        b[i] = b1;
        b[N + i] = b2;
    }
}

// Heun stage of the deformation gradient (deriv.cuh).  With k_dcol over all four planes a step is 4
// launches; 8 separate gradients and a pointwise kernel per stage were 26.  det F, displacement and
// labels at 512^2, nt = 32: 5640 -> 1390 us.
template <int LOGL>
__global__ void __launch_bounds__(256, 1) k_defgrad_row(DefGradStage a, int N, int lines, const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    defgrad_row_body<LOGL>(a, (uint32_t)N, lines, sm, tw, pdl_entry);
}

// grad f in one launch: blocks [0, tiles1) write d_1 f, the others d_2 f (both only read f).  Small
// calls are bound by the launches (64^2: three launches 8.7 us, one 4.3 us).
struct GradArgs {
    DColArgs col;
    ColMap m;
    float* out2;
    int log1, log2, tiles1, npairs, lines;
};
__global__ void __launch_bounds__(128) k_grad(GradArgs a, const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    if ((int)blockIdx.x < a.tiles1) {
        DISPATCH_LOG(a.log1, dcol_body<LG, 10 - LG, true>(a.col, a.m, blockIdx.x, sm, tw, pdl_entry));
    } else {
        DISPATCH_LOG(a.log2, drow_body<LG, false>(a.col.f, nullptr, a.out2, blockIdx.x - a.tiles1, a.lines, a.npairs, sm,
                                                  tw, pdl_entry));
    }
}

// out += d_2 f, out written by the preceding column kernel (the divergence)
template <int LOGL>
__global__ void __launch_bounds__(128) k_add_d2(const float* f, float* out, int npairs, int lines,
                                                const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    drow_body<LOGL, true>(f, out, out, blockIdx.x, lines, npairs, sm, tw, pdl_entry);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// columns per block of the column kernels as a template parameter: C L / 8 threads, 32 to 256 (16 on a 16 x 16 grid)
template <int LG, typename F>
static void dispatch_cols(int C, F&& f) {
    const int lt = LG - 3;  // log2 threads of one column
    int lc = 0;
    while ((1 << lc) < C) ++lc;
    switch (lc + lt) {
        case 4: if constexpr (4 - lt >= 0) f(std::integral_constant<int, 4 - lt>()); break;
        case 5: if constexpr (5 - lt >= 0) f(std::integral_constant<int, 5 - lt>()); break;
        case 6: if constexpr (6 - lt >= 0) f(std::integral_constant<int, 6 - lt>()); break;
        case 7: if constexpr (7 - lt >= 0) f(std::integral_constant<int, 7 - lt>()); break;
        case 8: if constexpr (8 - lt >= 0) f(std::integral_constant<int, 8 - lt>()); break;
        default: break;
    }
}

// out = d_1 (f mul [+ f2 mul2]) (mul nullable) for nb fields bs floats apart
void launch_dcol(reg_ctx* ctx, const DColArgs& a, int nb, long long bs) {
    const int L = ctx->n1, W = ctx->n2 / 2, C = cols_per_cta(ctx);
    int lw = 0;
    while ((1 << lw) < W) ++lw;
    const ColMap m{lw, 0, W, W};
    const size_t smem = dcol_smem(C, L);
    ktimer_begin(ctx, KC_COL, 4.0 * nb * (2 + (a.mul ? 1 : 0) + (a.f2 ? 2 : 0)) * ctx->N);
    DISPATCH_LOG(ctx->log1, dispatch_cols<LG>(C, [&](auto lc) {
        auto kern = k_dcol<LG, decltype(lc)::value>;
        set_smem(kern, smem);
        launch_k(ctx, kern, dim3(W / C, nb), C * (L / 8), smem, a, m, bs, ctx->tw);
    }));
    ktimer_end(ctx);
}

// row kernels of the transport: R rows = R / 2 pairs a block
struct PairCfg { int lines, threads, grid; size_t smem; bool pre; };
static PairCfg pair_cfg(reg_ctx* ctx) {
    PairCfg c;
    c.lines = rows_per_cta(ctx) / 2;
    c.threads = c.lines * (ctx->n2 / 8);
    c.grid = ctx->n1 / 2 / c.lines;
    c.smem = drow_smem(c.lines, ctx->n2);
    c.pre = prefetch_rows(ctx);
    return c;
}

void launch_row_adv(reg_ctx* ctx, const AdvStage<2>& a, int nb) {
    const PairCfg g = pair_cfg(ctx);
    // floats per node: u_s 1, u_j 1 (stage 2), D 1, v 2, u_out 1, source 1 or 4 (+ 1 stored), grad_out 2
    const double fl = (a.zero ? 0 : 2) + (a.stage == 2 && a.uj ? 1 : 0) + (a.u_out ? 3 : 0) + (a.src_in ? 1 : 0) +
                      (a.gm ? 4 : 0) + (a.src_out ? 1 : 0) + (a.grad_out ? 2 : 0);
    ktimer_begin(ctx, KC_ROWSTAGE, 4.0 * fl * nb * ctx->N);
    DISPATCH_LOG(ctx->log2, {
        auto kern = (g.pre || LG == 10) ? k_adv_row<LG, true> : k_adv_row<LG, (LG == 10)>;
        set_smem(kern, g.smem);
        launch_k(ctx, kern, dim3(g.grid, nb), g.threads, g.smem, a, ctx->N, g.lines, ctx->tw);
    });
    ktimer_end(ctx);
}

void launch_row_adj(reg_ctx* ctx, const AdjStage<2>& a) {
    const PairCfg g = pair_cfg(ctx);
    // lam_s 1, lam_j 1 (stage 2), D 1, v_2 1, l_out 1, body force b read + write 4 and gm 2; full Newton:
    // lam_src 1, v~_2 1, grad m~ 2 (stage 2)
    const double fl = 4 + (a.stage == 2 ? 1 : 0) + (a.b ? 6 : 0) + (a.lsrc ? 2 + (a.b ? 2 : 0) : 0);
    ktimer_begin(ctx, KC_ROWSTAGE, 4.0 * fl * ctx->N);
    DISPATCH_LOG(ctx->log2, {
        auto kern = a.lsrc ? k_adj_row<LG, false, true>
                           : ((g.pre || LG == 10) ? k_adj_row<LG, true, false> : k_adj_row<LG, (LG == 10), false>);
        set_smem(kern, g.smem);
        launch_k(ctx, kern, g.grid, g.threads, g.smem, a, ctx->N, g.lines, ctx->tw);
    });
    ktimer_end(ctx);
}

void launch_adj_init(reg_ctx* ctx, const float* a, float ca, const float* c, float cb, float* lam, float* b,
                     const float* gm, float w, const float* lsrc, const float* gmt) {
    // a 1 (optional), c 1, lam 1, b 2 + gm 2; full Newton: lsrc 1, grad m~ 2
    ktimer_begin(ctx, KC_POINT, 4.0 * ((a ? 1 : 0) + 6 + (lsrc ? 3 : 0)) * ctx->N);
    launch_k(ctx, k_adj_init, NBLK_RED, NTHREADS, 0, a, ca, c, cb, lam, b, gm, w, lsrc, gmt, ctx->N);
    ktimer_end(ctx);
}

void launch_defgrad_stage(reg_ctx* ctx, const DefGradStage& a) {
    const PairCfg g = pair_cfg(ctx);
    // F 4, F* 4 (stage 2), D 4, gv 4, v 2, out 4
    ktimer_begin(ctx, KC_ROWSTAGE, 4.0 * (18 + (a.stage == 2 ? 4 : 0)) * ctx->N);
    DISPATCH_LOG(ctx->log2, {
        auto kern = k_defgrad_row<LG>;
        set_smem(kern, g.smem);
        launch_k(ctx, kern, dim3(ctx->n1 / g.lines, 2), g.threads, g.smem, a, ctx->N, g.lines, ctx->tw);
    });
    ktimer_end(ctx);
}

// 128 threads a block whatever the axis lengths: 1024 / n1 columns, 1024 / n2 pairs of rows
void launch_grad(reg_ctx* ctx, const float* f, float* out) {
    const int W = ctx->n2 / 2, C = 1024 / ctx->n1;
    GradArgs a;
    a.col = DColArgs{f, nullptr, nullptr, nullptr, out};
    a.m = ColMap{ctx->log2 - 1, 0, W, W};
    a.out2 = out + ctx->N;
    a.log1 = ctx->log1;
    a.log2 = ctx->log2;
    a.tiles1 = (W + C - 1) / C;
    a.npairs = ctx->n1 / 2;
    a.lines = 1024 / ctx->n2;
    const int tiles2 = (a.npairs + a.lines - 1) / a.lines;
    ktimer_begin(ctx, KC_ROW, 16.0 * ctx->N);
    launch_k(ctx, k_grad, a.tiles1 + tiles2, 128, dcol_smem(C, ctx->n1), a, ctx->tw);
    ktimer_end(ctx);
}

void launch_add_d2(reg_ctx* ctx, const float* f, float* out) {
    const int npairs = ctx->n1 / 2, lines = 1024 / ctx->n2;
    ktimer_begin(ctx, KC_ROW, 12.0 * ctx->N);
    DISPATCH_LOG(ctx->log2, launch_k(ctx, k_add_d2<LG>, (npairs + lines - 1) / lines, 128, drow_smem(lines, ctx->n2), f,
                                     out, npairs, lines, ctx->tw));
    ktimer_end(ctx);
}
