// Whole transport solves in one launch for grids of 64 to 256 points per axis (Heun's RK2 of the
// state, adjoint, incremental state and incremental adjoint equations of Mang & Biros, arXiv
// 1503.00757, Sec. 3), resident in a thread-block cluster.
//
// On these grids a stage's two launches (transport.cu) cost about 4 us and compute for a fraction
// of it.  Here a cluster of CS CTAs owns the grid, R = n1 / CS rows each; u_j, the velocity and the
// body force live in registers for the whole solve, and a stage is
//   publish the stage's field in shared memory -> cluster barrier (meanwhile: x^2 derivative of the
//   own rows) -> x^1 derivative of C = n2 / (2 CS) packed columns, gathered from the row owners'
//   shared memory and scattered back to it -> cluster barrier -> update in registers.
// The transforms, the products and their order are those of transport.cu (deriv.cuh), so the
// results are the same bit for bit.  Half the threads are the row role, half the column role, so the
// two derivatives of a stage run side by side (one role doing both: 231 us for the gradient at
// 128^2, nt = 16; two roles: 208; kernel pairs: 318).  Bound by the latency of one transform pair
// and two cluster barriers a stage, about 2.3 us.  At 256^2 the 16 SMs of the largest cluster compute
// as long as the kernel pairs wait (302 against 301 us a matvec, nt = 16), so the line is below it.
// Matvecs, nt = 16, us each, resident against pairs, for one solve and for 32 at once: 64^2 103 / 213
// and 5.4 / 28.7, 64 x 256 119 / 275 and 11.7 / 29.6, 256 x 64 146 / 252 and 14.7 / 29.8, 128^2 135 /
// 277 and 13.6 / 30.6, 128 x 256 160 / 285 and 22.4 / 31.0, 256 x 128 178 / 279 and 26.2 / 31.5.
#include <map>
#include <mutex>

#include "cluster.cuh"
#include "deriv.cuh"
#include "internal.h"
#include "launch.cuh"

namespace {

template <int LOG1, int LOG2>
struct RsGeom {
    static constexpr int N1 = 1 << LOG1, N2 = 1 << LOG2, N = N1 * N2;
    static constexpr int CS = N >= 16384 ? 16 : 8;   // CTAs of the cluster
    static constexpr int R = N1 / CS;                // rows of a CTA
    static constexpr int PR = R / 2;                 // pairs of rows
    static constexpr int C = N2 / 2 / CS;            // packed columns of a CTA
    static constexpr int T1 = N1 / 8, T2 = N2 / 8;   // threads of a column / of a pair of rows
    static constexpr int TB = PR * T2;               // threads of the row role; = C T1, of the column role
    static constexpr size_t SMEM = (size_t)2 * R * N2 * sizeof(float) +
                                   (2 * (size_t)PR * (N2 + N2 / 8) + 2 * (size_t)C * (N1 + N1 / 8)) * sizeof(float2);
    static_assert(TB == C * T1 && TB >= 32 && TB <= 128 && R % 2 == 0, "the two roles have the same size, whole warps");
};

template <int LOG1, int LOG2, int MODE>
__global__ void __launch_bounds__(2 * RsGeom<LOG1, LOG2>::TB, 1) k_resident(RsArgs a, const float2* __restrict__ tw) {
    using G = RsGeom<LOG1, LOG2>;
    constexpr int N = G::N, N2 = G::N2, T2 = G::T2, C = G::C, R = G::R;
    extern __shared__ __align__(16) float2 sm[];
    float* U = reinterpret_cast<float*>(sm);   // field whose x^1 derivative is taken, own rows
    float* D = U + R * N2;                     // that derivative, own rows
    float2* Xr = reinterpret_cast<float2*>(D + R * N2);
    float2* Xc = Xr + 2 * G::PR * fft_buf(N2);
    const int rank = (int)cl_rank();
    const int nt = a.nt;
    if ((int)threadIdx.x >= G::TB) {
        // ---------------- column role: x^1 derivatives of the published fields ----------------
        const int id = threadIdx.x - G::TB, c = id & (C - 1), tc = id / C;  // column, rows tc + k T1
        LineTw<LOG1, true> W;
        W.load(tw, tc);
        float2 *cur = Xc + c, *nxt = cur + C * fft_buf(G::N1);
        // row tc + k T1 is row tc % R of CTA tc / R + k CS / 8
        const int owner = tc / R, off = (tc - owner * R) * N2 + 2 * (rank * C + c);
        uint32_t from[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) from[k] = cl_map(U + off, owner + k * (G::CS / 8));
        constexpr uint32_t UD = R * N2 * sizeof(float);  // D follows U in every CTA
        pdl_entry();
        const int stages = MODE == RS_STATE ? 2 * nt + 1 : (MODE == RS_ADJOINT ? 2 * nt : 4 * nt - 1);
#pragma unroll 1
        for (int s = 0; s < stages; ++s) {
            cl_arrive();
            cl_wait();
            float2 d[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) d[k] = cl_load(from[k]);
            line_deriv<LOG1, C>(d, tc, cur, nxt, [] { asm volatile("bar.sync 1, %0;" ::"n"(G::TB) : "memory"); }, W);
#pragma unroll
            for (int k = 0; k < 8; ++k) cl_store(from[k] + UD, d[k]);
            cl_arrive();
            cl_wait();
        }
        return;
    }
    // ---------------- row role: the fields, x^2 derivatives and updates ----------------
    const int q = threadIdx.x / T2, t = threadIdx.x - q * T2;    // pair of rows, entry t + k T2
    const uint32_t g0 = (uint32_t)(rank * R + 2 * q) * N2 + t;   // own entries in a global field
    const int s0 = 2 * q * N2 + t;                               // and in U, D
    LineTw<LOG2, true> Wr;
    Wr.load(tw, t);
    float2 *rcur = Xr + 2 * q * fft_buf(N2), *rnxt = rcur + fft_buf(N2);
    pdl_entry();
    auto pair = [&](const float* p, int k) { return make_float2(p[g0 + k * T2], p[g0 + N2 + k * T2]); };
    auto put = [&](float* p, int k, float2 w) { p[g0 + k * T2] = w.x; p[g0 + N2 + k * T2] = w.y; };
    // x <- d_2 x; d <- d_1 of the field whose own rows are f.  `between` runs while the columns are at work.
    auto derivs = [&](const float2 (&f)[8], float2 (&x)[8], float2 (&d)[8], auto&& between) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            U[s0 + k * T2] = f[k].x;
            U[s0 + N2 + k * T2] = f[k].y;
        }
        cl_arrive();
        line_deriv<LOG2, 1>(x, t, rcur, rnxt, RowSync<LOG2>(), Wr);
        cl_wait();
        cl_arrive();
        between();
        cl_wait();
#pragma unroll
        for (int k = 0; k < 8; ++k) d[k] = make_float2(D[s0 + k * T2], D[s0 + N2 + k * T2]);
    };
    float2 v1[8], v2[8], u[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        v1[k] = pair(a.v, k);
        v2[k] = pair(a.v + N, k);
        u[k] = MODE == RS_STATE ? pair(a.m0, k) : make_float2(0.f, 0.f);
    }
    if constexpr (MODE != RS_ADJOINT) {
        float2 us[8], src[8], x[8], d[8];
        auto source = [&](int j) {  // -v~ . grad m(t_j)
            const float* gm = a.gm + (size_t)j * 2 * N;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                float2 s = make_float2(0.f, 0.f);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float2 w = pair(a.vt + e * N, k), g = pair(gm + e * N, k);
                    s = make_float2(fmaf(-w.x, g.x, s.x), fmaf(-w.y, g.y, s.y));
                }
                src[k] = s;
            }
        };
        // u_j + c (E + h k), E = 0 (stage 1) or u* - u_j
        auto update = [&](float2 (&out)[8], bool second) {
            const float cc = second ? 0.5f : 1.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                float2 E = second ? csub(us[k], u[k]) : make_float2(0.f, 0.f);
                if (MODE == RS_MATVEC) E = make_float2(fmaf(a.h, src[k].x, E.x), fmaf(a.h, src[k].y, E.y));
                const float2 w2 = cscale(v2[k], -a.h), w1 = cscale(v1[k], -a.h);
                E = make_float2(fmaf(w2.x, x[k].x, E.x), fmaf(w2.y, x[k].y, E.y));
                E = make_float2(fmaf(w1.x, d[k].x, E.x), fmaf(w1.y, d[k].y, E.y));
                out[k] = make_float2(fmaf(cc, E.x, u[k].x), fmaf(cc, E.y, u[k].y));
            }
        };
        auto keep_grad = [&](int j) {
            float* gm = a.gm_out + (size_t)j * 2 * N;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                put(gm, k, d[k]);
                put(gm + N, k, x[k]);
            }
        };
        if (MODE == RS_MATVEC) source(0);
#pragma unroll 1
        for (int j = 0; j < nt; ++j) {
            if (MODE == RS_MATVEC && j == 0) {  // m~(0) = 0
#pragma unroll
                for (int k = 0; k < 8; ++k) us[k] = make_float2(a.h * src[k].x, a.h * src[k].y);
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) x[k] = u[k];
                derivs(u, x, d, [] {});
                if (MODE == RS_STATE) keep_grad(j);
                update(us, false);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = us[k];
            derivs(us, x, d, [&] { if (MODE == RS_MATVEC) source(j + 1); });
            update(u, true);
        }
        if (MODE == RS_STATE) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                x[k] = u[k];
                put(a.m_out, k, u[k]);
            }
            derivs(u, x, d, [] {});
            keep_grad(nt);
        }
    }
    if constexpr (MODE != RS_STATE) {
        float2 b1[8], b2[8], x[8], f[8], d[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float2 l;
            if (MODE == RS_MATVEC) {  // lam~(1) = -m~(1)
                l = make_float2(-u[k].x, -u[k].y);
            } else {
                const float2 p = pair(a.adj_c, k), r = pair(a.adj_a, k);
                l = make_float2(fmaf(a.ca, r.x, a.cb * p.x), fmaf(a.ca, r.y, a.cb * p.y));
            }
            u[k] = l;
            const float w = 0.5f * a.h;
            const float2 ga = pair(a.gm + (size_t)nt * 2 * N, k), gb = pair(a.gm + (size_t)nt * 2 * N + N, k);
            b1[k] = make_float2(__fmul_rn(w * l.x, ga.x), __fmul_rn(w * l.y, ga.y));
            b2[k] = make_float2(__fmul_rn(w * l.x, gb.x), __fmul_rn(w * l.y, gb.y));
        }
#pragma unroll 1
        for (int j = nt; j >= 1; --j) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                x[k] = make_float2(__fmul_rn(u[k].x, v2[k].x), __fmul_rn(u[k].y, v2[k].y));
                f[k] = make_float2(__fmul_rn(u[k].x, v1[k].x), __fmul_rn(u[k].y, v1[k].y));
            }
            derivs(f, x, d, [] {});
            float2 ls[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float2 dv = cadd(x[k], d[k]);
                ls[k] = make_float2(fmaf(a.h, dv.x, 0.f) + u[k].x, fmaf(a.h, dv.y, 0.f) + u[k].y);
                x[k] = make_float2(__fmul_rn(ls[k].x, v2[k].x), __fmul_rn(ls[k].y, v2[k].y));
                f[k] = make_float2(__fmul_rn(ls[k].x, v1[k].x), __fmul_rn(ls[k].y, v1[k].y));
            }
            const float w = j == 1 ? 0.5f * a.h : a.h;
            const float* gm = a.gm + (size_t)(j - 1) * 2 * N;
            float2 ga[8], gb[8];
            derivs(f, x, d, [&] {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    ga[k] = pair(gm, k);
                    gb[k] = pair(gm + N, k);
                }
            });
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float2 dv = cadd(x[k], d[k]), e = csub(ls[k], u[k]);
                u[k].x = fmaf(0.5f, fmaf(a.h, dv.x, e.x), u[k].x);
                u[k].y = fmaf(0.5f, fmaf(a.h, dv.y, e.y), u[k].y);
                const float2 l = cscale(u[k], w);
                b1[k] = make_float2(fmaf(l.x, ga[k].x, b1[k].x), fmaf(l.y, ga[k].y, b1[k].y));
                b2[k] = make_float2(fmaf(l.x, gb[k].x, b2[k].x), fmaf(l.y, gb[k].y, b2[k].y));
            }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            put(a.b, k, b1[k]);
            put(a.b + N, k, b2[k]);
        }
    }
}

template <int LOG1, int LOG2, int MODE>
cudaLaunchConfig_t rs_config(cudaStream_t st, cudaLaunchAttribute* attr, bool pdl) {
    using G = RsGeom<LOG1, LOG2>;
    return cluster_config(G::CS, 2 * G::TB, G::SMEM, st, attr, pdl);
}

template <int LOG1, int LOG2, int MODE>
bool rs_prepare() {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = rs_config<LOG1, LOG2, MODE>(0, attr, false);
    return cluster_prepare(k_resident<LOG1, LOG2, MODE>, cfg);
}

}  // namespace

bool rs_available(int log1, int log2) {
    if (log1 < 6 || log1 > 8 || log2 < 6 || log2 > 8 || log1 + log2 > 15) return false;
    static std::mutex mu;
    static std::map<int, bool> known;  // per device and grid: the attributes apply to the current device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> lock(mu);
    const int key = dev * 256 + log1 * 16 + log2;
    auto it = known.find(key);
    if (it != known.end()) return it->second;
    bool ok = false;
    RS_DISPATCH(log1, log2, ok = rs_prepare<B1, B2, RS_STATE>() && rs_prepare<B1, B2, RS_ADJOINT>() &&
                                 rs_prepare<B1, B2, RS_MATVEC>());
    return known[key] = ok;
}

void launch_resident(reg_ctx* ctx, int mode, const RsArgs& a) {
    // fields once per time level they are used at, as for the cluster kernel (transport_cluster.cu)
    const double fields = mode == RS_STATE ? 3 + 1 + 2.0 * (a.nt + 1)
                                           : (mode == RS_ADJOINT ? 6 + 2.0 * (a.nt + 1) : 6 + 4.0 * (a.nt + 1));
    ktimer_begin(ctx, KC_TRANSPORT, 4.0 * fields * ctx->N);
    RS_DISPATCH(ctx->log1, ctx->log2, {
        cudaLaunchAttribute attr[2];
        if (mode == RS_STATE) {
            cudaLaunchConfig_t cfg = rs_config<B1, B2, RS_STATE>(ctx->stream, attr, ctx->pdl);
            launch_cfg<RsArgs, const float2*>(ctx->build, cfg, k_resident<B1, B2, RS_STATE>, a, ctx->tw);
        } else if (mode == RS_ADJOINT) {
            cudaLaunchConfig_t cfg = rs_config<B1, B2, RS_ADJOINT>(ctx->stream, attr, ctx->pdl);
            launch_cfg<RsArgs, const float2*>(ctx->build, cfg, k_resident<B1, B2, RS_ADJOINT>, a, ctx->tw);
        } else {
            cudaLaunchConfig_t cfg = rs_config<B1, B2, RS_MATVEC>(ctx->stream, attr, ctx->pdl);
            launch_cfg<RsArgs, const float2*>(ctx->build, cfg, k_resident<B1, B2, RS_MATVEC>, a, ctx->tw);
        }
    });
    ktimer_end(ctx);
}
