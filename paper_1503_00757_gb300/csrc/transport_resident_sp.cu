// The spectral RK2 stages of kernels.cu (k_row_adv_sp, k_row_adj_sp and the OP_GRAD1 / OP_DIV1
// column passes) resident in a thread-block cluster: whole transport solves of the H2 and H3
// problems on grids of 64 to 256 points per axis, up to 2^14 points, in one launch.
//
// Those problems keep the spectral stages because their Krylov iteration amplifies a change of
// rounding (kernels.cu), so this kernel does their arithmetic, expression by expression (products
// and FMAs spelled out where the compiler contracts differently around another memory layout),
// and the results are the same bit for bit.  Only where the data lives differs: a cluster of CS CTAs owns
// R = n1 / CS rows each, whose fields, velocity and body force stay in registers and whose row
// spectra stay in shared memory; the column pass gathers its C = n2 / (2 CS) columns from the row
// owners over distributed shared memory and scatters the result back (two cluster barriers a
// stage instead of two launches of about 9 us together at 128^2; eight mixed 128^2 pairs, two
// Newton steps each: 13.5 to 16 ms with the launches, 8.2 to 9.5 ms).  Bound by latency, like transport_resident.cu.
#include <map>
#include <mutex>

#include "cluster.cuh"
#include "fft.cuh"
#include "fft_reg.cuh"
#include "internal.h"
#include "launch.cuh"

namespace {

template <int LOG1, int LOG2>
struct SpGeom {
    static constexpr int N1 = 1 << LOG1, N2 = 1 << LOG2, N = N1 * N2, W = N2 / 2;
    static constexpr int CS = N >= 16384 ? 16 : 8;
    static constexpr int R = N1 / CS;                // rows of a CTA (a multiple of 4: whole spectrum tiles)
    static constexpr int C = W / CS;                 // spectrum columns of a CTA
    static constexpr int T1 = N1 / 8, T2 = N2 / 8;   // threads of a column / of a row
    static constexpr int THREADS = R * T2;           // = 2 C T1: one row per T2 threads
    static constexpr size_t ENTRIES = (size_t)4 * R * W + 2 * (size_t)R * (N2 + N2 / 8) + 2 * (size_t)C * (N1 + N1 / 8) + N1;
    static constexpr size_t SMEM = ENTRIES * sizeof(float2);
    static_assert(THREADS == 2 * C * T1 && R % 4 == 0 && THREADS <= 256, "rows and columns share the threads");
};

template <int LOG1, int LOG2, int MODE>
__global__ void __launch_bounds__(SpGeom<LOG1, LOG2>::THREADS, 1) k_resident_sp(RsArgs a, const float2* __restrict__ tw) {
    using G = SpGeom<LOG1, LOG2>;
    constexpr int N = G::N, L = G::N2, W = G::W, T = G::T2, R = G::R, C = G::C, L1 = G::N1, T1 = G::T1, H1 = L1 / 2;
    extern __shared__ __align__(16) float2 sm[];
    float2* S1 = sm;              // row spectra of the stage's field (adjoint: of the x^1 flux), tiled (sp_idx)
    float2* S2 = S1 + R * W;      // of the x^2 flux
    float2* Gd = S2 + R * W;      // result of the column pass
    float2* Z = Gd + R * W;       // R rows of real values, then R / 2 full spectra
    float2* Xr = Z + R * W;
    float2* Xc = Xr + 2 * R * fft_buf(L);
    float2* Zs = Xc + 2 * C * fft_buf(L1);  // column 0's spectrum
    float* O = reinterpret_cast<float*>(Z);
    const int rank = (int)cl_rank();
    const int q = threadIdx.x / T, t = threadIdx.x - q * T;   // row, entry t + k T
    const size_t rowbase = (size_t)(rank * R + q) * L;
    // column role of the first C T1 threads: column c, rows tc + k T1 (row tc % R of CTA tc / R + k CS / 8)
    const bool colact = (int)threadIdx.x < C * T1;
    const int c = threadIdx.x % C, tc = threadIdx.x / C;
    const int e = rank * C + c;
    const int owner = tc / R, off = (int)sp_idx(tc - owner * R, e, W);
    const float scale = 1.0f / (float)N;
    uint32_t from[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) from[k] = colact ? cl_map(S1 + off, owner + k * (G::CS / 8)) : 0u;
    constexpr uint32_t SP_PLANE = R * W * sizeof(float2);  // S2 and Gd follow S1 in every CTA
    pdl_entry();

    float2* xb = Xr + 2 * q * fft_buf(L);
    // forward transform of the rows in O (two rows per transform) and their packed spectra into S1
    auto rows_forward = [&]() {
        const bool act2 = q < R / 2;
        float2 x[8];
        if (act2) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int j = t + k * T;
                x[k] = make_float2(O[2 * q * L + j], O[(2 * q + 1) * L + j]);
            }
        }
        reg_fft<LOG2, false>(x, t, act2, xb, xb + fft_buf(L), tw);
        if (act2) {
#pragma unroll
            for (int k = 0; k < 8; ++k) Z[q * L + t + k * T] = x[k];
        }
        __syncthreads();
        for (int idx = threadIdx.x; idx < R * W; idx += blockDim.x) {
            const int r = ((idx / (4 * W)) << 2) | (idx & 3);
            const int ee = (idx >> 2) & (W - 1);
            S1[idx] = split_entry<LOG2>(Z + (r >> 1) * L, r & 1, ee);
        }
    };
    // flux spectra of x (one row per transform) into S1, S2; the R full spectra take Gd and Z, both
    // consumed by then
    auto flux_forward = [&](float2 (&x)[8]) {
        reg_fft<LOG2, false>(x, t, true, xb, xb + fft_buf(L), tw);
#pragma unroll
        for (int k = 0; k < 8; ++k) Gd[q * L + t + k * T] = x[k];
        __syncthreads();
        for (int idx = threadIdx.x; idx < R * W; idx += blockDim.x) {
            const int r = ((idx / (4 * W)) << 2) | (idx & 3);
            const int ee = (idx >> 2) & (W - 1);
            S1[idx] = split_entry<LOG2>(Gd + r * L, 0, ee);
            S2[idx] = split_entry<LOG2>(Gd + r * L, 1, ee);
        }
    };
    // Gd <- i k1~ S1 / N along x^1 (DIV: plus (i k2~ / n2) S2), as k_col<OP_GRAD1 / OP_DIV1>
    auto column = [&](bool div) {
        cl_arrive();
        cl_wait();
        float2 x[8];
        if (colact) {
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = cl_load(from[k]);
        }
        float2* cb = Xc + 2 * c * fft_buf(L1);
        reg_fft<LOG1, false>(x, tc, colact, cb, cb + fft_buf(L1), tw);
        if (rank == 0) {
            if (colact && c == 0) {
#pragma unroll
                for (int k = 0; k < 8; ++k) Zs[tc + k * T1] = x[k];
            }
            __syncthreads();
        }
        if (colact) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int p = tc + k * T1;
                const float k1 = (p < H1) ? (float)p : (float)(p - L1);
                const float k1o = (p == H1) ? 0.f : k1;
                if (e > 0) {
                    const float w = __fmul_rn(k1o, scale);
                    x[k] = make_float2(__fmul_rn(-x[k].y, w), __fmul_rn(x[k].x, w));
                } else {
                    const int pm = (L1 - p) & (L1 - 1);
                    const float2 zp = x[k], zm = Zs[pm];
                    const float2 xv = make_float2(0.5f * (zp.x + zm.x), 0.5f * (zp.y - zm.y));
                    const float2 xh = make_float2(0.5f * (zp.y + zm.y), -0.5f * (zp.x - zm.x));
                    const float2 yv = cscale(cmuli(xv), k1o * scale), yb = cscale(cmuli(xh), k1o * scale);
                    x[k] = make_float2(yv.x - yb.y, yv.y + yb.x);
                }
            }
        }
        __syncthreads();
        reg_fft<LOG1, true>(x, tc, colact, cb, cb + fft_buf(L1), tw);
        if (colact) {
            const float cd2 = 1.0f / (float)L;
            const float ce = cd2 * (float)e;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                float2 val = x[k];
                if (div) {
                    const float2 f2 = cl_load(from[k] + SP_PLANE);
                    val = make_float2(val.x - ce * f2.y, val.y + ce * f2.x);
                }
                cl_store(from[k] + 2 * SP_PLANE, val);
            }
        }
        cl_arrive();
        cl_wait();
    };

    float pv1[8], pv2[8], u[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const size_t idx = rowbase + t + k * T;
        pv1[k] = a.v[idx];
        pv2[k] = a.v[N + idx];
        u[k] = MODE == RS_STATE ? a.m0[idx] : 0.f;
    }
    const int nt = a.nt;
    if constexpr (MODE != RS_ADJOINT) {
        float us[8], psrc[8];
        if (MODE == RS_STATE) {
#pragma unroll
            for (int k = 0; k < 8; ++k) O[q * L + t + k * T] = u[k];
            __syncthreads();
            rows_forward();
        }
#pragma unroll 1
        for (int s = 0; s < 2 * nt; ++s) {
            const int j = s >> 1, stage = 1 + (s & 1);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                psrc[k] = 0.f;
                if (MODE == RS_MATVEC) {
                    const size_t idx = rowbase + t + k * T;
                    const float* gm = a.gm + (size_t)(j + stage - 1) * 2 * N;
                    psrc[k] = -(a.vt[idx] * gm[idx] + a.vt[N + idx] * gm[N + idx]);
                }
            }
            float2 x[8];
            if (MODE == RS_MATVEC && s == 0) {
#pragma unroll
                for (int k = 0; k < 8; ++k) x[k] = make_float2(0.f, 0.f);
            } else {
                column(false);
                const float cc = 1.0f / (float)L;
#pragma unroll
                for (int k = 0; k < 8; ++k) x[k] = merged_entry_d2<LOG2>(Gd, q, S1, q, t + k * T, cc);
                reg_fft<LOG2, true>(x, t, true, xb, xb + fft_buf(L), tw);
            }
            const float hh = a.h;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const size_t idx = rowbase + t + k * T;
                const float d1 = x[k].x, d2 = x[k].y;
                if (MODE == RS_STATE && stage == 1) {
                    float* gm = a.gm_out + (size_t)j * 2 * N;
                    gm[idx] = d1;
                    gm[N + idx] = d2;
                }
                const float kk = psrc[k] - fmaf(pv1[k], d1, __fmul_rn(pv2[k], d2));
                const float pus = stage == 2 ? us[k] : 0.f;
                const float out = (stage == 1) ? fmaf(hh, kk, u[k]) : 0.5f * fmaf(hh, kk, u[k] + pus);
                if (stage == 1) us[k] = out;
                else u[k] = out;
                O[q * L + t + k * T] = out;
            }
            if (MODE == RS_MATVEC && s == 2 * nt - 1) break;
            __syncthreads();
            rows_forward();
        }
        if (MODE == RS_STATE) {
            // m(1) and its row spectra, from which the caller takes grad m(1)
#pragma unroll
            for (int k = 0; k < 8; ++k) a.m_out[rowbase + t + k * T] = u[k];
            __syncthreads();
            for (int idx = threadIdx.x; idx < R * W; idx += blockDim.x) a.s_out[(size_t)rank * R * W + idx] = S1[idx];
        }
    }
    if constexpr (MODE != RS_STATE) {
        float b1[8], b2[8], ls[8];
        float2 x[8];
        {
            const float w = 0.5f * a.h;
            const float* gm = a.gm + (size_t)nt * 2 * N;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const size_t idx = rowbase + t + k * T;
                float l;
                if (MODE == RS_MATVEC) {
                    l = -1.f * u[k];
                } else {
                    l = a.cb * a.adj_c[idx];
                    l = fmaf(a.ca, a.adj_a[idx], l);
                }
                u[k] = l;
                b1[k] = w * l * gm[idx];
                b2[k] = w * l * gm[N + idx];
                x[k] = make_float2(__fmul_rn(l, pv1[k]), __fmul_rn(l, pv2[k]));
            }
        }
        flux_forward(x);
#pragma unroll 1
        for (int s = 0; s < 2 * nt; ++s) {
            const int j = nt - (s >> 1), stage = 1 + (s & 1);
            const float* gm = a.gm + (size_t)(j - 1) * 2 * N;
            float ga[8], gb[8];
            if (stage == 2) {  // fetched while the columns are at work
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const size_t idx = rowbase + t + k * T;
                    ga[k] = gm[idx];
                    gb[k] = gm[N + idx];
                }
            }
            column(true);
            const bool act1 = q < R / 2;
            if (act1) {
#pragma unroll
                for (int k = 0; k < 8; ++k) x[k] = merged_entry<LOG2>(Gd, 2 * q, Gd, 2 * q + 1, t + k * T);
            }
            reg_fft<LOG2, true>(x, t, act1, xb, xb + fft_buf(L), tw);
            if (act1) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    O[2 * q * L + t + k * T] = x[k].x;
                    O[(2 * q + 1) * L + t + k * T] = x[k].y;
                }
            }
            __syncthreads();
            const float w = (j - 1 == 0) ? 0.5f * a.h : a.h;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float dv = O[q * L + t + k * T];
                const float pls = stage == 2 ? ls[k] : 0.f;
                const float out = (stage == 1) ? fmaf(a.h, dv, u[k]) : 0.5f * fmaf(a.h, dv, u[k] + pls);
                if (stage == 2) {
                    const float wl = w * out;
                    b1[k] = fmaf(wl, ga[k], b1[k]);
                    b2[k] = fmaf(wl, gb[k], b2[k]);
                    u[k] = out;
                } else {
                    ls[k] = out;
                }
                x[k] = make_float2(__fmul_rn(out, pv1[k]), __fmul_rn(out, pv2[k]));
            }
            if (s == 2 * nt - 1) break;
            flux_forward(x);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const size_t idx = rowbase + t + k * T;
            a.b[idx] = b1[k];
            a.b[N + idx] = b2[k];
        }
    }
}

template <int LOG1, int LOG2, int MODE>
cudaLaunchConfig_t sp_config(cudaStream_t st, cudaLaunchAttribute* attr, bool pdl) {
    using G = SpGeom<LOG1, LOG2>;
    return cluster_config(G::CS, G::THREADS, G::SMEM, st, attr, pdl);
}

template <int LOG1, int LOG2, int MODE>
bool sp_prepare() {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = sp_config<LOG1, LOG2, MODE>(0, attr, false);
    return cluster_prepare(k_resident_sp<LOG1, LOG2, MODE>, cfg);
}

}  // namespace

bool rs_sp_available(int log1, int log2) {
    // 2^15 points: faster alone (matvec, nt = 16: 393 us against 449 at 256 x 128, 459 against 564 at
    // 128 x 256) but not with many solves at once, whose clusters take turns on the chip: 8 solves 83
    // against 79 us each, 32 solves 61 against 39 (128 x 256: 96 against 91, 70 against 36).  On 2^14
    // points it is ahead at every number of solves: 128 x 128 alone 314 against 538, 32 at once 30.0
    // against 30.9.
    if (log1 < 6 || log1 > 8 || log2 < 6 || log2 > 8 || log1 + log2 > 14) return false;
    static std::mutex mu;
    static std::map<int, bool> known;  // per device and grid: the attributes apply to the current device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> lock(mu);
    const int key = dev * 256 + log1 * 16 + log2;
    auto it = known.find(key);
    if (it != known.end()) return it->second;
    bool ok = false;
    RS_SP_DISPATCH(log1, log2, ok = sp_prepare<B1, B2, RS_STATE>() && sp_prepare<B1, B2, RS_ADJOINT>() &&
                                 sp_prepare<B1, B2, RS_MATVEC>());
    return known[key] = ok;
}

void launch_resident_sp(reg_ctx* ctx, int mode, const RsArgs& a) {
    const double fields = mode == RS_STATE ? 3 + 1 + 2.0 * (a.nt + 1)
                                           : (mode == RS_ADJOINT ? 6 + 2.0 * (a.nt + 1) : 6 + 4.0 * (a.nt + 1));
    ktimer_begin(ctx, KC_TRANSPORT, 4.0 * fields * ctx->N);
    RS_SP_DISPATCH(ctx->log1, ctx->log2, {
        cudaLaunchAttribute attr[2];
        if (mode == RS_STATE) {
            cudaLaunchConfig_t cfg = sp_config<B1, B2, RS_STATE>(ctx->stream, attr, ctx->pdl);
            launch_cfg<RsArgs, const float2*>(ctx->build, cfg, k_resident_sp<B1, B2, RS_STATE>, a, ctx->tw);
        } else if (mode == RS_ADJOINT) {
            cudaLaunchConfig_t cfg = sp_config<B1, B2, RS_ADJOINT>(ctx->stream, attr, ctx->pdl);
            launch_cfg<RsArgs, const float2*>(ctx->build, cfg, k_resident_sp<B1, B2, RS_ADJOINT>, a, ctx->tw);
        } else {
            cudaLaunchConfig_t cfg = sp_config<B1, B2, RS_MATVEC>(ctx->stream, attr, ctx->pdl);
            launch_cfg<RsArgs, const float2*>(ctx->build, cfg, k_resident_sp<B1, B2, RS_MATVEC>, a, ctx->tw);
        }
    });
    ktimer_end(ctx);
}
