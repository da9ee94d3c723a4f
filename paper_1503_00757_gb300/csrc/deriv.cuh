// Spectral first derivatives along one axis of a real field, and the pieces the transport
// kernels build from them (pseudospectral discretization, Sec. 4 of Mang & Biros).
//
// d/dx_a of a real field is a one-dimensional operation: transform along axis a, multiply by
// i k~ (odd symbol, Nyquist entry zero), transform back.  The transforms along the other axes
// cancel, so no multi-dimensional spectrum is ever formed.  i k~ is the symbol of a real
// operator, so two real lines travel as the real and imaginary part of one complex line and
// come back as their two derivatives, with no splitting or merging in between:
//   * along a strided axis the two lines are neighbours in the contiguous direction, so a
//     float2 load of the field is the packed pair ("column" of float2);
//   * along the contiguous axis the two lines are two rows (or one row of two fields).
// Length-L lines use the radix-8 register transform of fft_reg.cuh (T = L / 8 threads, 8
// values each); the exchange-buffer layout and the barrier are the caller's.
#pragma once
#include <cuda_runtime.h>

#include "fft.cuh"
#include "fft_reg.cuh"

// shared-memory exchanges of one length-2^logl transform
__host__ __device__ constexpr int fft_exchanges(int logl) { return logl % 3 == 0 ? logl / 3 - 1 : logl / 3; }

// A thread's twiddles of every pass, loaded once (before the wait on the preceding kernel: the
// table is constant) and used by the forward transform and, conjugated, by the inverse.
template <int LOGL>
struct LineTw {
    static constexpr int NP = tw_passes(LOGL);
    float2 w[NP > 0 ? NP : 1][7];
    __device__ __forceinline__ void load(const float2* __restrict__ tw, int t) {
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int k = 1; k < 8; ++k)
                w[i][k - 1] = __ldg(&tw[twp_base(LOGL) + tw_off(LOGL, i) + (k - 1) * tw_groups(LOGL, i) + (t >> (3 * i))]);
    }
};

// The transform of reg_fft (same passes, same arithmetic) with the caller's exchange layout:
// idx(pos) is the buffer index of line position pos, sync() the barrier over the line's threads.
// Exchanges alternate between two buffers; `nxt` is written next and swapped with `cur` after
// each exchange, so consecutive transforms need no barrier in between: when a buffer is written
// again, the barrier of the exchange through the other one lies after its last reads.
template <int LOGL, bool INV, class Idx, class Sync>
__device__ __forceinline__ void line_fft(float2 (&x)[8], int t, float2*& cur, float2*& nxt, Idx idx, Sync sync,
                                         const LineTw<LOGL>& W) {
    constexpr int L = 1 << LOGL, T = L >> 3, NP8 = LOGL / 3, REM = LOGL - 3 * NP8;
#pragma unroll
    for (int i = 0; i < NP8; ++i) {
        const int ls = 3 * i, s = 1 << ls, q = t & (s - 1), p = t >> ls, m = L >> (ls + 3);
        const bool last = (i == NP8 - 1) && (REM == 0);
        if (i > 0) {
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = cur[idx(q + s * (p + k * m))];
        }
        dft8<INV>(x);
        if (!last) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                float2 y = x[k];
                if (k > 0) {
                    float2 w = W.w[i][k - 1];
                    if (INV) w.y = -w.y;
                    y = cmul(y, w);
                }
                nxt[idx(q + s * (8 * p + k))] = y;
            }
            sync();
            float2* b = cur; cur = nxt; nxt = b;
        }
    }
    if (REM == 1) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 a = cur[idx(t + j * T)], b = cur[idx(t + j * T + 4 * T)];
            x[j] = cadd(a, b);
            x[j + 4] = csub(a, b);
        }
    } else if (REM == 2) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int q = t + j * T;
            const float2 a0 = cur[idx(q)], a1 = cur[idx(q + 2 * T)], a2 = cur[idx(q + 4 * T)], a3 = cur[idx(q + 6 * T)];
            const float2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = mul_mi<INV>(csub(a1, a3));
            x[j] = cadd(t0, t2);
            x[j + 2] = cadd(t1, t3);
            x[j + 4] = csub(t0, t2);
            x[j + 6] = csub(t1, t3);
        }
    }
}

// x <- d/dx of the complex line whose entries t + k T are x[k]
template <int LOGL, class Idx, class Sync>
__device__ __forceinline__ void line_deriv(float2 (&x)[8], int t, float2*& cur, float2*& nxt, Idx idx, Sync sync,
                                           const LineTw<LOGL>& W) {
    constexpr int L = 1 << LOGL, T = L >> 3, H = L >> 1;
    line_fft<LOGL, false>(x, t, cur, nxt, idx, sync, W);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int p = t + k * T;
        const float kk = (p < H) ? (float)p : ((p == H) ? 0.f : (float)(p - L));
        x[k] = cscale(cmuli(x[k]), kk * (1.0f / (float)L));
    }
    line_fft<LOGL, true>(x, t, cur, nxt, idx, sync, W);
}

// ---- strided axis: columns of float2 ----
// Column l (0 <= l < ncols) starts at float2 index (l >> lq) * P + (l & ((1 << lq) - 1)); its
// entries are S apart.  2-D: lq covers all columns.  3-D axis 1: the same with n2 n3 / 2 columns;
// axis 2: lq = log2(n3 / 2), P = n2 n3 / 2, S = n3 / 2.
struct ColMap {
    int lq;
    int P;
    int S;
    int ncols;
};

// derivative of f (mul == nullptr), of f mul, or of f mul + f2 mul2, into out.  A CTA of
// C (L / 8) threads takes C neighbouring columns, the column index fastest over the threads: a
// load or store of one line position is C * 8 contiguous bytes, and in the exchange buffers
// (position-major, one padding position per 8) the 16 lanes of a 64-bit shared-memory access
// fall on distinct banks for every C >= 2.
struct DColArgs {
    const float* f;
    const float* mul;
    const float* f2;
    const float* mul2;
    float* out;
};

template <int LOGL, class Wait>
__device__ __forceinline__ void dcol_body(const DColArgs& a, const ColMap& m, int C, int lc, int tile, float2* sm,
                                          const float2* __restrict__ tw, Wait wait) {
    constexpr int L = 1 << LOGL, T = L >> 3;
    const int c = threadIdx.x & (C - 1), t = threadIdx.x >> lc;
    const int l = tile * C + c;
    const bool on = l < m.ncols;
    const size_t base = (size_t)(l >> m.lq) * m.P + (l & ((1 << m.lq) - 1));
    LineTw<LOGL> W;
    W.load(tw, t);
    float2 x[8];
    wait();
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = make_float2(0.f, 0.f);
    if (on) {
        const float2* f = reinterpret_cast<const float2*>(a.f) + base;
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = f[(size_t)(t + k * T) * m.S];
        if (a.mul) {
            const float2* g = reinterpret_cast<const float2*>(a.mul) + base;
            float2 y[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) y[k] = g[(size_t)(t + k * T) * m.S];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = make_float2(x[k].x * y[k].x, x[k].y * y[k].y);
            if (a.f2) {
                const float2* f2 = reinterpret_cast<const float2*>(a.f2) + base;
                const float2* g2 = reinterpret_cast<const float2*>(a.mul2) + base;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const size_t i = (size_t)(t + k * T) * m.S;
                    const float2 p = f2[i], q = g2[i];
                    x[k] = make_float2(fmaf(p.x, q.x, x[k].x), fmaf(p.y, q.y, x[k].y));
                }
            }
        }
    }
    float2* cur = sm + C * fft_buf(L);
    float2* nxt = sm;
    line_deriv<LOGL>(x, t, cur, nxt, [&](int pos) { return (fft_pad(pos) << lc) + c; }, [] { __syncthreads(); }, W);
    if (on) {
        float2* o = reinterpret_cast<float2*>(a.out) + base;
#pragma unroll
        for (int k = 0; k < 8; ++k) o[(size_t)(t + k * T) * m.S] = x[k];
    }
}

// shared memory of dcol_body: two exchange buffers of C columns
inline size_t dcol_smem(int C, int L) { return 2 * (size_t)C * fft_buf(L) * sizeof(float2); }

// ---- contiguous axis: pairs of rows ----
// barrier over the T = L / 8 threads of a row line: lines of up to 256 points lie in one warp
template <int LOGL>
struct RowSync {
    __device__ __forceinline__ void operator()() const {
        if (LOGL <= 8) __syncwarp();
        else __syncthreads();
    }
};

template <int LOGL>
__device__ __forceinline__ void row_deriv(float2 (&x)[8], int t, int q, float2* sm, const LineTw<LOGL>& W) {
    constexpr int L = 1 << LOGL;
    float2* cur = sm + 2 * q * fft_buf(L);
    float2* nxt = cur + fft_buf(L);
    line_deriv<LOGL>(x, t, cur, nxt, [](int pos) { return fft_pad(pos); }, RowSync<LOGL>(), W);
}
inline size_t drow_smem(int lines, int L) { return 2 * (size_t)lines * fft_buf(L) * sizeof(float2); }

// ---- transport stages along the contiguous axis ----
// DIM = 2 or 3 space dimensions; D[a] holds the derivative along strided axis a (from the
// preceding column kernel), the derivative along the last axis is taken here.  Vector fields are
// DIM planes of N.
//
// Heun stage of the state and incremental state equations (Eq. (e:state-eq-elim),
// (e:inc-state-eq-elim)):  k = -v . grad u_s + src, src = -v~ . grad m(t);
//   stage 1: u* = u_j + h k;  stage 2: u_{j+1} = (u_j + u* + h k) / 2.
// A source time t_{j+1} serves stage 2 of step j and stage 1 of step j + 1, so stage 2 stores
// src (src_out) and the next stage 1 reads that one plane (src_in) instead of 2 DIM planes.
template <int DIM>
struct AdvRow {
    const float* D[DIM - 1];
    const float* uj;      // u_j; nullptr: u_j = 0
    const float* us;      // stage 2: u*.  (stage 1 differentiates u_j)
    const float* v;
    const float* src_in;  // nullable
    const float* gm;      // nullable: src = -vt . gm
    const float* vt;
    float* src_out;       // nullable
    float* u_out;         // nullable (gradient only)
    float* grad_out;      // nullable: grad u_s (DIM planes)
    float h;
    int stage;
    int late;             // 1: read every operand after the wait (one may come from the launch just before)
    int zero;             // 1: u_s = 0, no derivative (D unused)
    size_t bs;            // blockIdx.y: field stride of uj, us, D, src_in, u_out
};

// Heun stage of the adjoint equation, backward in time (Eq. (e:adj-eq-elim),
// (e:inc-adj-eq-elim)):  k = div(lam_s v) with D[a] = d_a(lam_s v_a);
//   stage 1: lam* = lam_j + h k;  stage 2: lam_{j-1} = (lam_j + lam* + h k) / 2 and
//   b += w lam_{j-1} grad m_{j-1}.
// Full Newton (lsrc != nullptr): the flux is lam_s v + lsrc vt and b += w lsrc gmt.
template <int DIM>
struct AdjRow {
    const float* D[DIM - 1];
    const float* lj;
    const float* ls;      // stage 2: lam*
    const float* v;
    float* l_out;
    float* b;             // stage 2
    const float* gm;
    float w;
    float h;
    int stage;
    const float* lsrc;
    const float* vt;
    const float* gmt;
};

// One thread holds entries t + k T of rows 2 q and 2 q + 1 (x[k].x, x[k].y).  PRE: the row
// derivative and everything that does not depend on D are computed before the wait on the column
// kernel (u_s was written two launches back), so only the D loads, one FMA per strided axis and
// the stores follow it.  That is the point of the split: the row transforms leave the critical
// path of the launch chain.
// Rounding: the increment E = h k (stage 2: (u* - u_j) + h k) is summed on its own, at its own
// magnitude, and added to u_j once, so a stage rounds u a single time (what it rounds off is
// white noise that every later derivative multiplies by k).
template <int LOGL, int DIM, bool PRE, class Wait>
__device__ __forceinline__ void adv_row_body(const AdvRow<DIM>& a, size_t N, int lines, float2* sm,
                                             const float2* __restrict__ tw, Wait wait) {
    constexpr int L = 1 << LOGL, T = L >> 3;
    const int q = threadIdx.x / T, t = threadIdx.x - q * T;
    const size_t r0 = ((size_t)blockIdx.x * lines + q) * 2 * L + t, r1 = r0 + L;
    const size_t bo = blockIdx.y * a.bs;
    const bool early = PRE && !a.late;
    LineTw<LOGL> W;
    if (!a.zero) W.load(tw, t);
    if (!early) wait();
    float2 x[8], u[8], E[8], hv[DIM - 1][8];
    const float* us = (a.stage == 2 ? a.us : a.uj);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int j = k * T;
        u[k] = a.uj ? make_float2(a.uj[bo + r0 + j], a.uj[bo + r1 + j]) : make_float2(0.f, 0.f);
        x[k] = u[k];
        if (a.stage == 2) x[k] = make_float2(us[bo + r0 + j], us[bo + r1 + j]);
        E[k] = csub(x[k], u[k]);
    }
    if (a.u_out) {
        if (a.src_in) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int j = k * T;
                E[k].x = fmaf(a.h, a.src_in[bo + r0 + j], E[k].x);
                E[k].y = fmaf(a.h, a.src_in[bo + r1 + j], E[k].y);
            }
        } else if (a.gm) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int j = k * T;
                float2 s = make_float2(0.f, 0.f);
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    s.x = fmaf(-a.vt[d * N + r0 + j], a.gm[d * N + r0 + j], s.x);
                    s.y = fmaf(-a.vt[d * N + r1 + j], a.gm[d * N + r1 + j], s.y);
                }
                if (a.src_out) {
                    a.src_out[r0 + j] = s.x;
                    a.src_out[r1 + j] = s.y;
                }
                E[k].x = fmaf(a.h, s.x, E[k].x);
                E[k].y = fmaf(a.h, s.y, E[k].y);
            }
        }
        if (PRE) {
#pragma unroll
            for (int d = 0; d < DIM - 1; ++d)
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    hv[d][k] = make_float2(-a.h * a.v[d * N + r0 + k * T], -a.h * a.v[d * N + r1 + k * T]);
        }
    }
    if (!a.zero) {
        row_deriv<LOGL>(x, t, q, sm, W);
        if (a.u_out) {
            const float* vl = a.v + (DIM - 1) * N;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                E[k].x = fmaf(-a.h * vl[r0 + k * T], x[k].x, E[k].x);
                E[k].y = fmaf(-a.h * vl[r1 + k * T], x[k].y, E[k].y);
            }
        }
    }
    if (early) wait();
    float2 D[DIM - 1][8];
    if (!a.zero) {
#pragma unroll
        for (int d = 0; d < DIM - 1; ++d)
#pragma unroll
            for (int k = 0; k < 8; ++k) D[d][k] = make_float2(a.D[d][bo + r0 + k * T], a.D[d][bo + r1 + k * T]);
    }
    if (a.grad_out) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
#pragma unroll
            for (int d = 0; d < DIM - 1; ++d) {
                a.grad_out[d * N + r0 + k * T] = a.zero ? 0.f : D[d][k].x;
                a.grad_out[d * N + r1 + k * T] = a.zero ? 0.f : D[d][k].y;
            }
            a.grad_out[(DIM - 1) * N + r0 + k * T] = a.zero ? 0.f : x[k].x;
            a.grad_out[(DIM - 1) * N + r1 + k * T] = a.zero ? 0.f : x[k].y;
        }
    }
    if (a.u_out) {
        if (!PRE && !a.zero) {
#pragma unroll
            for (int d = 0; d < DIM - 1; ++d)
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    hv[d][k] = make_float2(-a.h * a.v[d * N + r0 + k * T], -a.h * a.v[d * N + r1 + k * T]);
        }
        const float c = a.stage == 2 ? 0.5f : 1.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (!a.zero) {
#pragma unroll
                for (int d = 0; d < DIM - 1; ++d) {
                    E[k].x = fmaf(hv[d][k].x, D[d][k].x, E[k].x);
                    E[k].y = fmaf(hv[d][k].y, D[d][k].y, E[k].y);
                }
            }
            a.u_out[bo + r0 + k * T] = fmaf(c, E[k].x, u[k].x);
            a.u_out[bo + r1 + k * T] = fmaf(c, E[k].y, u[k].y);
        }
    }
}

template <int LOGL, int DIM, bool PRE, bool FULL, class Wait>
__device__ __forceinline__ void adj_row_body(const AdjRow<DIM>& a, size_t N, int lines, float2* sm,
                                             const float2* __restrict__ tw, Wait wait) {
    constexpr int L = 1 << LOGL, T = L >> 3;
    const int q = threadIdx.x / T, t = threadIdx.x - q * T;
    const size_t r0 = ((size_t)blockIdx.x * lines + q) * 2 * L + t, r1 = r0 + L;
    LineTw<LOGL> W;
    W.load(tw, t);
    if (!PRE) wait();
    float2 x[8], u[8], E[8];
    const float* vl = a.v + (DIM - 1) * N;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int j = k * T;
        u[k] = make_float2(a.lj[r0 + j], a.lj[r1 + j]);
        float2 s = u[k];
        if (a.stage == 2) s = make_float2(a.ls[r0 + j], a.ls[r1 + j]);
        E[k] = csub(s, u[k]);
        x[k] = make_float2(s.x * vl[r0 + j], s.y * vl[r1 + j]);
        if (FULL) {
            const float* tl = a.vt + (DIM - 1) * N;
            x[k].x = fmaf(a.lsrc[r0 + j], tl[r0 + j], x[k].x);
            x[k].y = fmaf(a.lsrc[r1 + j], tl[r1 + j], x[k].y);
        }
    }
    row_deriv<LOGL>(x, t, q, sm, W);
    if (PRE) wait();
    float2 D[DIM - 1][8];
#pragma unroll
    for (int d = 0; d < DIM - 1; ++d)
#pragma unroll
        for (int k = 0; k < 8; ++k) D[d][k] = make_float2(a.D[d][r0 + k * T], a.D[d][r1 + k * T]);
    const float c = a.stage == 2 ? 0.5f : 1.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float2 dv = x[k];
#pragma unroll
        for (int d = 0; d < DIM - 1; ++d) dv = cadd(dv, D[d][k]);
        u[k].x = fmaf(c, fmaf(a.h, dv.x, E[k].x), u[k].x);
        u[k].y = fmaf(c, fmaf(a.h, dv.y, E[k].y), u[k].y);
        a.l_out[r0 + k * T] = u[k].x;
        a.l_out[r1 + k * T] = u[k].y;
    }
    if (!a.b) return;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        float2 b[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const size_t i0 = d * N + r0 + k * T, i1 = d * N + r1 + k * T;
            b[k] = make_float2(fmaf(a.w * u[k].x, a.gm[i0], a.b[i0]), fmaf(a.w * u[k].y, a.gm[i1], a.b[i1]));
            if (FULL) {
                b[k].x = fmaf(a.w * a.lsrc[r0 + k * T], a.gmt[i0], b[k].x);
                b[k].y = fmaf(a.w * a.lsrc[r1 + k * T], a.gmt[i1], b[k].y);
            }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            a.b[d * N + r0 + k * T] = b[k].x;
            a.b[d * N + r1 + k * T] = b[k].y;
        }
    }
}
