// Autotuner of the FFT tile choices.  The row kernels process R
// grid rows per CTA and the column kernels C columns per CTA, and the
// RK2 row kernels either prefetch their operands before waiting on the
// preceding kernel (P = 1, more registers) or load them after the FFT (P = 0,
// two 512-thread CTAs per SM).  The best choice depends on the grid (CTA count
// against the 152 SMs, threads and shared memory per CTA) and on how many
// solves share the GPU, so it is found by timing the Gauss-Newton Hessian
// matvec (the incremental state and adjoint transports, Algorithm 2) for
// every valid (R, C, P) with a given number of solves running concurrently on
// their own streams, each with and without programmatic dependent launch
// (D): early launch hides one solve's launch latency but lets waiting CTAs
// hold SM resources, and which wins depends on the concurrency.
//
// What is timed is what contexts run: the axis-wise stages of H1 problems and
// the spectral stages of H2 and H3 problems are different kernels with
// different needs, so each kind has its own entry, timed with a context of that
// kind; where the transport solves are resident (small grids), R, C and D are
// those of the kernels around them, and P, which no kernel reads then, keeps
// its default.  The cluster-resident transport kernel of reg_set_transport is
// not a candidate: measured on a GB300 it is slower than the kernel pairs at
// every grid size, nt and concurrency tried.  Results live in a process-wide
// table per (device, n1, n2, kind); contexts created afterwards on that device
// and grid use them.
#include <cmath>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "internal.h"

namespace {
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int, int>, Tuned> g_tune;

bool pow2_grid(int n) { return n >= 16 && n <= 1024 && (n & (n - 1)) == 0; }

struct Lane {
    reg_ctx* ctx = nullptr;
    cudaStream_t st = nullptr;
    cudaEvent_t done = nullptr;
};

// Milliseconds per Hessian matvec (throughput over `lanes.size()` concurrent
// solves, linearized already) with the choice t; < 0 on failure.
double time_matvec(const Tuned& t, size_t n2, std::vector<Lane>& lanes, const float* v, float* out, cudaStream_t root,
                   cudaEvent_t e0, cudaEvent_t e1) {
    bool ok = true;
    for (size_t i = 0; ok && i < lanes.size(); ++i) {
        Lane& L = lanes[i];
        const bool valid = tiles_valid(L.ctx->n1, L.ctx->n2, t.R, t.C, t.P);  // else the default rule's
        ok = reg_set_tiles(L.ctx, valid ? t.R : 0, valid ? t.C : 0, t.P) == REG_OK && reg_set_pdl(L.ctx, t.D) == REG_OK;
        for (int k = 0; ok && k < 2; ++k) ok = reg_hessian_matvec(L.ctx, v, out + i * n2) == REG_OK;
    }
    const int reps = 4;
    double ms = -1.0;
    for (size_t i = 0; ok && i < lanes.size(); ++i) ok = cudaStreamSynchronize(lanes[i].st) == cudaSuccess;
    if (ok) ok = cudaEventRecord(e0, root) == cudaSuccess;
    for (size_t i = 0; ok && i < lanes.size(); ++i) {
        Lane& L = lanes[i];
        ok = cudaStreamWaitEvent(L.st, e0, 0) == cudaSuccess;
        for (int k = 0; ok && k < reps; ++k) ok = reg_hessian_matvec(L.ctx, v, out + i * n2) == REG_OK;
        if (ok) ok = cudaEventRecord(L.done, L.st) == cudaSuccess && cudaStreamWaitEvent(root, L.done, 0) == cudaSuccess;
    }
    float dt = 0.f;
    if (ok && cudaEventRecord(e1, root) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess &&
        cudaEventElapsedTime(&dt, e0, e1) == cudaSuccess)
        ms = dt / (reps * (double)lanes.size());
    for (Lane& L : lanes) cudaStreamSynchronize(L.st);
    return ms;
}
}  // namespace

bool tuned_tiles(int dev, int n1, int n2, TuneKind kind, Tuned* t) {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tune.find(std::make_tuple(dev, n1, n2, (int)kind));
    if (it == g_tune.end()) return false;
    *t = it->second;
    return true;
}

int autotune_kind(reg_grid grid, int nt, int concurrency, bool force, TuneKind kind, Tuned* out_t, double* out_ms) {
    if (!pow2_grid(grid.n1) || !pow2_grid(grid.n2))
        return reg_fail(REG_ERR_ARG, "n1 and n2 must be powers of two in [16, 1024]");
    if (nt < 1 || nt > 4096) return reg_fail(REG_ERR_ARG, "nt must be in [1, 4096]");
    if (concurrency < 1 || concurrency > 16) return reg_fail(REG_ERR_ARG, "concurrency must be in [1, 16]");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return reg_fail(REG_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (!force && tuned_tiles(dev, grid.n1, grid.n2, kind, out_t)) {
        if (out_ms) *out_ms = -1.0;
        return REG_OK;
    }
    const size_t N = (size_t)grid.n1 * grid.n2;
    const int K = concurrency;
    float* buf = nullptr;
    if (cudaMalloc(&buf, sizeof(float) * (4 + 2 * (size_t)K) * N) != cudaSuccess) {
        cudaGetLastError();
        return reg_fail(REG_ERR_NOMEM, "autotune buffers");
    }
    std::vector<Lane> lanes(K);
    cudaStream_t root = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int status = REG_OK;
    bool ok = cudaStreamCreateWithFlags(&root, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess;
    for (Lane& L : lanes)
        ok = ok && cudaStreamCreateWithFlags(&L.st, cudaStreamNonBlocking) == cudaSuccess &&
             cudaEventCreateWithFlags(&L.done, cudaEventDisableTiming) == cudaSuccess;
    // zero images and velocity: every kernel runs its full work, no value can overflow
    ok = ok && cudaMemsetAsync(buf, 0, sizeof(float) * (4 + 2 * (size_t)K) * N, root) == cudaSuccess &&
         cudaStreamSynchronize(root) == cudaSuccess;
    if (!ok) status = reg_fail(REG_ERR_CUDA, "autotune streams / events");
    float *mT = buf, *mR = buf + N, *v = buf + 2 * N, *out = buf + 4 * N;
    for (int i = 0; status == REG_OK && i < K; ++i) {
        Lane& L = lanes[i];
        status = reg_create(grid, nt, kind == TUNE_AXIS ? REG_H1 : REG_H2, 1e-3, INFINITY, 0.0, &L.ctx);
        if (status == REG_OK) status = reg_set_stream(L.ctx, L.st);
        if (status == REG_OK) status = reg_set_images(L.ctx, mT, mR);
        if (status == REG_OK) status = reg_gradient(L.ctx, v, out + i * 2 * N, nullptr);
    }
    int R0, C0, P0;
    default_tiles(grid.n1, grid.n2, &R0, &C0, &P0);
    std::vector<Tuned> cands;
    for (int r = 4; r <= grid.n1; r *= 2)
        for (int c = 2; c <= grid.n2 / 2; c *= 2)
            for (int p = 0; p <= 1; ++p)
                for (int d = 0; d <= 1; ++d)
                    if (tiles_valid(grid.n1, grid.n2, r, c, p) &&
                        (p == P0 || status != REG_OK || !resident_transport(lanes[0].ctx)))
                        cands.push_back(Tuned{r, c, p, d});
    if (cands.empty()) cands.push_back(Tuned{R0, C0, P0, 1});  // 16 x 16
    // two passes over all candidates, each candidate's faster time kept: neighbouring choices
    // differ by a few percent, about the run-to-run spread of one short measurement
    std::vector<double> tbest(cands.size(), -1.0);
    for (int pass = 0; pass < 2 && status == REG_OK; ++pass) {
        for (size_t i = 0; status == REG_OK && i < cands.size(); ++i) {
            const double ms = time_matvec(cands[i], 2 * N, lanes, v, out, root, e0, e1);
            if (ms < 0.0) {
                status = reg_fail(REG_ERR_CUDA, std::string("autotune candidate failed: ") + reg_last_error());
                break;
            }
            if (tbest[i] < 0.0 || ms < tbest[i]) tbest[i] = ms;
        }
    }
    double best = -1.0;
    Tuned choice = cands[0];
    for (size_t i = 0; status == REG_OK && i < cands.size(); ++i) {
        if (best < 0.0 || tbest[i] < best) {
            best = tbest[i];
            choice = cands[i];
        }
    }
    if (root) cudaStreamSynchronize(root);
    for (Lane& L : lanes) {
        if (L.st) cudaStreamSynchronize(L.st);
        if (L.ctx) reg_destroy(L.ctx);
        if (L.done) cudaEventDestroy(L.done);
        if (L.st) cudaStreamDestroy(L.st);
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (root) cudaStreamDestroy(root);
    cudaFree(buf);
    if (status != REG_OK) return status;
    {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        g_tune[std::make_tuple(dev, grid.n1, grid.n2, (int)kind)] = choice;
    }
    *out_t = choice;
    if (out_ms) *out_ms = best;
    return REG_OK;
}

extern "C" int reg_autotune(reg_grid grid, int nt, int concurrency, int force, int* rows_per_cta, int* cols_per_cta,
                            int* prefetch, int* pdl, double* ms_per_matvec) {
    Tuned t, spectral;
    int st = autotune_kind(grid, nt, concurrency, force != 0, TUNE_AXIS, &t, ms_per_matvec);
    if (st == REG_OK) st = autotune_kind(grid, nt, concurrency, force != 0, TUNE_SPECTRAL, &spectral, nullptr);
    if (st != REG_OK) return st;
    if (rows_per_cta) *rows_per_cta = t.R;
    if (cols_per_cta) *cols_per_cta = t.C;
    if (prefetch) *prefetch = t.P;
    if (pdl) *pdl = t.D;
    return REG_OK;
}

extern "C" int reg_tile_config(reg_ctx* ctx, int* rows_per_cta, int* cols_per_cta, int* prefetch, int* pdl) {
    if (!ctx) return reg_fail(REG_ERR_ARG, "ctx is NULL");
    int R, C, P;
    default_tiles(ctx->n1, ctx->n2, &R, &C, &P);
    const bool set = ctx->tileR > 0;
    if (rows_per_cta) *rows_per_cta = set ? ctx->tileR : R;
    if (cols_per_cta) *cols_per_cta = set ? ctx->tileC : C;
    if (prefetch) *prefetch = set ? ctx->tileP : P;
    if (pdl) *pdl = ctx->pdl ? 1 : 0;
    return REG_OK;
}
