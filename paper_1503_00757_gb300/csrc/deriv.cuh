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

#include <cstdint>

#include "fft.cuh"
#include "fft_reg.cuh"

// shared-memory exchanges of one length-2^logl transform
__host__ __device__ constexpr int fft_exchanges(int logl) { return logl % 3 == 0 ? logl / 3 - 1 : logl / 3; }

// Twiddles of a thread.  REG: loaded into registers once, before the wait on the preceding kernel
// (the table is constant), for the forward transform and, conjugated, the inverse: nothing but the
// data is fetched on the critical path of a launch chain.  Otherwise read from the table (L1) where
// they are used: up to 28 registers fewer, for kernels that live on warps in flight.
template <int LOGL, bool REG>
struct LineTw {
    static constexpr int NP = tw_passes(LOGL);
    float2 w[REG && NP > 0 ? NP : 1][7];
    const float2* tab;
    __device__ __forceinline__ void load(const float2* __restrict__ tw, int t) {
        if (REG) {
#pragma unroll
            for (int i = 0; i < NP; ++i)
#pragma unroll
                for (int k = 1; k < 8; ++k)
                    w[i][k - 1] = __ldg(&tw[twp_base(LOGL) + tw_off(LOGL, i) + (k - 1) * tw_groups(LOGL, i) + (t >> (3 * i))]);
        } else {
            tab = tw;
        }
    }
    __device__ __forceinline__ float2 get(int i, int k, int p) const {
        if (REG) return w[i][k - 1];
        return __ldg(&tab[twp_base(LOGL) + tw_off(LOGL, i) + (k - 1) * tw_groups(LOGL, i) + p]);
    }
};

// Exchange-buffer addresses of a line whose position p sits at (p + p / 8) M (+ the caller's base):
// one padding position per 8, M lines interleaved.  Every address is one base per pass plus a
// compile-time offset per k (a carry from t into the padding term cannot occur: in a write the
// k part is a multiple of 8 or below it, in a read k T is a multiple of 8 or t + k T mod 8 < 8),
// so the exchanges cost no integer arithmetic per element.
template <int LOGL, int M>
struct LineIdx {
    static constexpr int T = 1 << (LOGL - 3);
    template <int I>
    __device__ __forceinline__ static int wbase(int t) {  // pass I writes positions q + s (8 p + k)
        constexpr int s = 1 << (3 * I);
        const int q = t & (s - 1), p = t >> (3 * I);
        return (I == 0 ? 9 * p : q + (q >> 3) + 9 * s * p) * M;
    }
    template <int I>
    __host__ __device__ static constexpr int woff(int k) {
        return (I == 0 ? k : 9 * (1 << (3 * I)) / 8 * k) * M;
    }
    __device__ __forceinline__ static int rbase(int t) { return (T >= 8 ? t + (t >> 3) : t) * M; }  // position t + k T
    __host__ __device__ static constexpr int roff(int k) { return (T >= 8 ? k * (T + T / 8) : k * T + k * T / 8) * M; }
};

// In-register DFT of length 8; the odd outputs' factor sqrt(1/2) rides in the last additions.
template <bool INV>
__device__ __forceinline__ void line_dft8(float2 (&x)[8]) {
    const float r = 0.70710678118654752440f;
    const float2 b0 = cadd(x[0], x[4]), b1 = csub(x[0], x[4]);
    const float2 b2 = cadd(x[2], x[6]), b3 = mul_mi<INV>(csub(x[2], x[6]));
    const float2 b4 = cadd(x[1], x[5]), b5 = csub(x[1], x[5]);
    const float2 b6 = cadd(x[3], x[7]), b7 = mul_mi<INV>(csub(x[3], x[7]));
    const float2 E0 = cadd(b0, b2), E2 = csub(b0, b2), E1 = cadd(b1, b3), E3 = csub(b1, b3);
    const float2 O0 = cadd(b4, b6), O2 = mul_mi<INV>(csub(b4, b6)), O1 = cadd(b5, b7), O3 = csub(b5, b7);
    // w1 O1 = r (1 -/+ i) O1, w3 O3 = r (-1 -/+ i) O3
    const float2 p = INV ? make_float2(O1.x - O1.y, O1.x + O1.y) : make_float2(O1.x + O1.y, O1.y - O1.x);
    const float2 m = INV ? make_float2(O3.x + O3.y, O3.y - O3.x) : make_float2(O3.x - O3.y, O3.x + O3.y);
    x[0] = cadd(E0, O0); x[4] = csub(E0, O0);
    x[1] = make_float2(fmaf(r, p.x, E1.x), fmaf(r, p.y, E1.y));
    x[5] = make_float2(fmaf(-r, p.x, E1.x), fmaf(-r, p.y, E1.y));
    x[2] = cadd(E2, O2); x[6] = csub(E2, O2);
    x[3] = make_float2(fmaf(-r, m.x, E3.x), fmaf(-r, m.y, E3.y));
    x[7] = make_float2(fmaf(r, m.x, E3.x), fmaf(r, m.y, E3.y));
}

// radix-8 pass I of line_fft and the ones after it
template <int LOGL, bool INV, int M, int I, class Sync, class Tw>
__device__ __forceinline__ void line_pass(float2 (&x)[8], int t, float2*& cur, float2*& nxt, Sync sync, const Tw& W) {
    using X = LineIdx<LOGL, M>;
    constexpr int NP8 = LOGL / 3, REM = LOGL - 3 * NP8;
    if constexpr (I < NP8) {
        if constexpr (I > 0) {
            const float2* c = cur + X::rbase(t);
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = c[X::roff(k)];
        }
        line_dft8<INV>(x);
        if constexpr (!(I == NP8 - 1 && REM == 0)) {
            float2* n = nxt + X::template wbase<I>(t);
            n[0] = x[0];
#pragma unroll
            for (int k = 1; k < 8; ++k) {
                float2 w = W.get(I, k, t >> (3 * I));
                if (INV) w.y = -w.y;
                n[X::template woff<I>(k)] = cmul(x[k], w);
            }
            sync();
            float2* b = cur; cur = nxt; nxt = b;
        }
        line_pass<LOGL, INV, M, I + 1>(x, t, cur, nxt, sync, W);
    }
}

// The register radix-8 Stockham transform of fft_reg.cuh with the caller's barrier (sync: over the
// line's T = L / 8 threads) and M interleaved lines per exchange buffer; cur and nxt point at this
// line's position 0.  On entry and exit x[k] is entry t + k T; unnormalized.  Exchanges alternate
// between two buffers; `nxt` is written next and swapped with `cur` after each exchange, so
// consecutive transforms need no barrier in between: when a buffer is written again, the barrier
// of the exchange through the other one lies after its last reads.
template <int LOGL, bool INV, int M, class Sync, class Tw>
__device__ __forceinline__ void line_fft(float2 (&x)[8], int t, float2*& cur, float2*& nxt, Sync sync, const Tw& W) {
    using X = LineIdx<LOGL, M>;
    constexpr int REM = LOGL % 3;
    line_pass<LOGL, INV, M, 0>(x, t, cur, nxt, sync, W);
    if (REM == 1) {
        const float2* c = cur + X::rbase(t);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 a = c[X::roff(j)], b = c[X::roff(j + 4)];
            x[j] = cadd(a, b);
            x[j + 4] = csub(a, b);
        }
    } else if (REM == 2) {
        const float2* c = cur + X::rbase(t);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 a0 = c[X::roff(j)], a1 = c[X::roff(j + 2)], a2 = c[X::roff(j + 4)], a3 = c[X::roff(j + 6)];
            const float2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = mul_mi<INV>(csub(a1, a3));
            x[j] = cadd(t0, t2);
            x[j + 2] = cadd(t1, t3);
            x[j + 4] = csub(t0, t2);
            x[j + 6] = csub(t1, t3);
        }
    }
}

// x <- d/dx of the complex line whose entries t + k T are x[k]
template <int LOGL, int M, class Sync, class Tw>
__device__ __forceinline__ void line_deriv(float2 (&x)[8], int t, float2*& cur, float2*& nxt, Sync sync, const Tw& W) {
    constexpr int L = 1 << LOGL, T = L >> 3;
    constexpr float s = 1.0f / (float)L;
    line_fft<LOGL, false, M>(x, t, cur, nxt, sync, W);
    const float f = (float)t * s;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        // k~ / L of entry t + k T: (t + k T) / L below L / 2, 0 at L / 2, (t + k T) / L - 1 above
        float kk = f + (k < 4 ? (float)(k * T) * s : (float)(k * T - L) * s);
        if (k == 4 && t == 0) kk = 0.f;
        x[k] = make_float2(__fmul_rn(-kk, x[k].y), __fmul_rn(kk, x[k].x));
    }
    line_fft<LOGL, true, M>(x, t, cur, nxt, sync, W);
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

template <int LOGL, int LC, bool TWREG, class Wait>
__device__ __forceinline__ void dcol_body(const DColArgs& a, const ColMap& m, int tile, float2* sm,
                                          const float2* __restrict__ tw, Wait wait) {
    constexpr int L = 1 << LOGL, T = L >> 3, C = 1 << LC;
    const int c = threadIdx.x & (C - 1), t = threadIdx.x >> LC;
    const int l = tile * C + c;
    const bool on = l < m.ncols;
    const uint32_t base = (uint32_t)(l >> m.lq) * m.P + (l & ((1 << m.lq) - 1)) + (uint32_t)t * m.S;
    const uint32_t step = (uint32_t)T * m.S;
    LineTw<LOGL, TWREG> W;
    W.load(tw, t);
    float2 x[8], y[8];
    // the factor (the velocity: written two or more launches back) is fetched ahead of the wait
    if (on && a.mul) {
        const float2* g = reinterpret_cast<const float2*>(a.mul) + base;
#pragma unroll
        for (int k = 0; k < 8; ++k) y[k] = g[k * step];
    }
    wait();
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = make_float2(0.f, 0.f);
    if (on) {
        const float2* f = reinterpret_cast<const float2*>(a.f) + base;
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = f[k * step];
        if (a.mul) {
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = make_float2(__fmul_rn(x[k].x, y[k].x), __fmul_rn(x[k].y, y[k].y));
            if (a.f2) {
                const float2* f2 = reinterpret_cast<const float2*>(a.f2) + base;
                const float2* g2 = reinterpret_cast<const float2*>(a.mul2) + base;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 p = f2[k * step], q = g2[k * step];
                    x[k] = make_float2(fmaf(p.x, q.x, x[k].x), fmaf(p.y, q.y, x[k].y));
                }
            }
        }
    }
    float2* cur = sm + C * fft_buf(L) + c;
    float2* nxt = sm + c;
    line_deriv<LOGL, C>(x, t, cur, nxt, [] { __syncthreads(); }, W);
    if (on) {
        float2* o = reinterpret_cast<float2*>(a.out) + base;
#pragma unroll
        for (int k = 0; k < 8; ++k) o[k * step] = x[k];
    }
}

// ---- 16 entries a thread: lines of 128 and 256 points with one exchange per transform ----
// On fields that fill the chip dcol_body is bound by shared memory (l1tex 78 % busy at 128^3): two
// exchanges per transform of such a line.  A thread with 16 entries needs one: a DFT of length 16
// over its entries t + k T (T = L / 16), the factors w^(t j), one exchange, then a DFT of length T
// over t.  Half the threads per line, so it is for grids that have blocks to spare.
template <bool INV>
__device__ __forceinline__ void line_dft4(float2& a0, float2& a1, float2& a2, float2& a3) {
    const float2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = mul_mi<INV>(csub(a1, a3));
    a0 = cadd(t0, t2);
    a1 = cadd(t1, t3);
    a2 = csub(t0, t2);
    a3 = csub(t1, t3);
}
template <bool INV>
__device__ __forceinline__ void line_dft16(float2 (&x)[16]) {
    // k = k1 + 4 k2, j = j2 + 4 j1: DFT-4 over k2, w16^(k1 j2), DFT-4 over k1
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) line_dft4<INV>(x[k1], x[k1 + 4], x[k1 + 8], x[k1 + 12]);
    const float c = 0.92387953251128675613f, s = 0.38268343236508977173f, r = 0.70710678118654752440f;
    const float2 w[10] = {{1.f, 0.f}, {c, -s}, {r, -r}, {s, -c}, {0.f, -1.f}, {0.f, 0.f}, {-r, -r}, {0.f, 0.f}, {0.f, 0.f}, {-c, s}};
#pragma unroll
    for (int j2 = 1; j2 < 4; ++j2)
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1) {
            if (j2 * k1 == 4) {
                x[k1 + 4 * j2] = mul_mi<INV>(x[k1 + 4 * j2]);
            } else {
                const float2 u = w[j2 * k1];
                x[k1 + 4 * j2] = cmul(x[k1 + 4 * j2], make_float2(u.x, INV ? -u.y : u.y));
            }
        }
    float2 y[16];
#pragma unroll
    for (int j2 = 0; j2 < 4; ++j2) {
        line_dft4<INV>(x[4 * j2], x[4 * j2 + 1], x[4 * j2 + 2], x[4 * j2 + 3]);
#pragma unroll
        for (int j1 = 0; j1 < 4; ++j1) y[j2 + 4 * j1] = x[4 * j2 + j1];
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = y[k];
}

template <int LOGL>
struct Wide {
    static constexpr int L = 1 << LOGL, T = L / 16, C = 128 / T;      // 128 threads: C columns
    static constexpr int P = C >= 16 ? T : T + 1;                     // pitch of a row j of the exchange (16 lanes of
                                                                      // an access fall on distinct banks)
    static constexpr size_t SMEM = 2 * (size_t)16 * P * C * sizeof(float2);
};

template <int LOGL, bool INV>
__device__ __forceinline__ void wide_fft(float2 (&x)[16], int t, float2* buf, const float2 (&w)[15]) {
    using G = Wide<LOGL>;
    constexpr int C = G::C, P = G::P;
    line_dft16<INV>(x);
    buf[t * C] = x[0];
#pragma unroll
    for (int j = 1; j < 16; ++j) buf[(j * P + t) * C] = cmul(x[j], make_float2(w[j - 1].x, INV ? -w[j - 1].y : w[j - 1].y));
    __syncthreads();
    if constexpr (LOGL == 8) {
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = buf[(t * P + k) * C];
        line_dft16<INV>(x);
    } else {  // T = 8: rows t and t + 8, whose outputs interleave
        float2 a[8], b[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            a[k] = buf[(t * P + k) * C];
            b[k] = buf[((t + 8) * P + k) * C];
        }
        line_dft8<INV>(a);
        line_dft8<INV>(b);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            x[2 * k] = a[k];
            x[2 * k + 1] = b[k];
        }
    }
}

// dcol_body (without the second product) for LOGL = 7, 8 and 128 threads a block
template <int LOGL, class Wait>
__device__ __forceinline__ void dcol_wide_body(const DColArgs& a, const ColMap& m, int tile, float2* sm,
                                               const float2* __restrict__ tw, Wait wait) {
    using G = Wide<LOGL>;
    constexpr int L = G::L, T = G::T, C = G::C;
    const int c = threadIdx.x & (C - 1), t = threadIdx.x / C;
    const int l = tile * C + c;
    const bool on = l < m.ncols;
    const uint32_t base = (uint32_t)(l >> m.lq) * m.P + (l & ((1 << m.lq) - 1)) + (uint32_t)t * m.S;
    const uint32_t step = (uint32_t)T * m.S;
    float2 w[15];
#pragma unroll
    for (int j = 1; j < 16; ++j) w[j - 1] = __ldg(&tw[t * j * (REG_TW_N / L)]);
    wait();
    float2 x[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = make_float2(0.f, 0.f);
    if (on) {
        const float2* f = reinterpret_cast<const float2*>(a.f) + base;
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = f[k * step];
        if (a.mul) {
            const float2* g = reinterpret_cast<const float2*>(a.mul) + base;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const float2 y = g[k * step];
                x[k] = make_float2(__fmul_rn(x[k].x, y.x), __fmul_rn(x[k].y, y.y));
            }
        }
    }
    wide_fft<LOGL, false>(x, t, sm + c, w);
    const float f = (float)t * (1.0f / (float)L);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        float kk = f + (k < 8 ? (float)(k * T) : (float)(k * T - L)) * (1.0f / (float)L);
        if (k == 8 && t == 0) kk = 0.f;
        x[k] = make_float2(__fmul_rn(-kk, x[k].y), __fmul_rn(kk, x[k].x));
    }
    wide_fft<LOGL, true>(x, t, sm + 16 * G::P * C + c, w);
    if (on) {
        float2* o = reinterpret_cast<float2*>(a.out) + base;
#pragma unroll
        for (int k = 0; k < 16; ++k) o[k * step] = x[k];
    }
}

// shared memory of dcol_body: two exchange buffers of C columns
inline size_t dcol_smem(int C, int L) { return 2 * (size_t)C * fft_buf(L) * sizeof(float2); }

// ---- contiguous axis: pairs of rows ----
// barrier over the T = L / 8 threads of a row line: lines of up to 256 points lie in one warp
template <int LOGL>
struct RowSync {
    __device__ __forceinline__ void operator()() const {
        if (LOGL > 8) __syncthreads();
        else if (blockDim.x >= 32) __syncwarp();
        else __syncwarp((1u << blockDim.x) - 1u);  // the whole of a 16 x 16 grid
    }
};

template <int LOGL, class Tw>
__device__ __forceinline__ void row_deriv(float2 (&x)[8], int t, int q, float2* sm, const Tw& W) {
    constexpr int L = 1 << LOGL;
    float2* cur = sm + 2 * q * fft_buf(L);
    float2* nxt = cur + fft_buf(L);
    line_deriv<LOGL, 1>(x, t, cur, nxt, RowSync<LOGL>(), W);
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
struct AdvStage {
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
    uint32_t bs;          // blockIdx.y: field stride of uj, us, D, src_in, u_out
    uint32_t gs;          // blockIdx.y: stride of grad_out
};

// Heun stage of the adjoint equation, backward in time (Eq. (e:adj-eq-elim),
// (e:inc-adj-eq-elim)):  k = div(lam_s v) with D[a] = d_a(lam_s v_a);
//   stage 1: lam* = lam_j + h k;  stage 2: lam_{j-1} = (lam_j + lam* + h k) / 2 and
//   b += w lam_{j-1} grad m_{j-1}.
// Full Newton (lsrc != nullptr): the flux is lam_s v + lsrc vt and b += w lsrc gmt.
template <int DIM>
struct AdjStage {
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

// One thread holds entries t + k T of rows 2 q and 2 q + 1 (x[k].x, x[k].y).
// PRE: the row derivative and everything that does not depend on D are computed before the wait on
// the column kernel (u_s was written two launches back), so only the D loads, one FMA per strided
// axis and the stores follow it.  That is the point of the split: the row transforms leave the
// critical path of the launch chain.  Otherwise everything follows the wait and the operands are
// loaded after the transform, BATCH entries at a time, which halves the registers: for fields
// that fill the chip, where warps in flight hide latency and not the overlap with one kernel.
// Both variants do the same arithmetic in the same order (products that feed an addition of a
// transform are kept from contraction), so results do not depend on the choice.
// Rounding: the increment E = h k (stage 2: (u* - u_j) + h k) is summed on its own, at its own
// magnitude, and added to u_j once, so a stage rounds u a single time (what it rounds off is
// white noise that every later derivative multiplies by k).
template <int LOGL, int DIM, bool PRE, int BATCH, class Wait>
__device__ __forceinline__ void adv_row_body(const AdvStage<DIM>& a, uint32_t N, int lines, float2* sm,
                                             const float2* __restrict__ tw, Wait wait) {
    constexpr int L = 1 << LOGL, T = L >> 3;
    const int q = threadIdx.x / T, t = threadIdx.x - q * T;
    const uint32_t r0 = (blockIdx.x * lines + q) * 2 * L + t, r1 = r0 + L;
    const uint32_t bo = blockIdx.y * a.bs, go = blockIdx.y * a.gs;
    const bool early = PRE && !a.late;
    const float c = a.stage == 2 ? 0.5f : 1.f;
    const float* us = (a.stage == 2 ? a.us : a.uj);
    auto pair = [&](const float* p, uint32_t o, int k) { return make_float2(p[o + r0 + k * T], p[o + r1 + k * T]); };
    auto put = [&](float* p, uint32_t o, int k, float2 w) { p[o + r0 + k * T] = w.x; p[o + r1 + k * T] = w.y; };
    // src of entry k, and its store for the next stage 1
    auto source = [&](int k) {
        float2 s = make_float2(0.f, 0.f);
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            const float2 w = pair(a.vt, d * N, k), g = pair(a.gm, d * N, k);
            s = make_float2(fmaf(-w.x, g.x, s.x), fmaf(-w.y, g.y, s.y));
        }
        return s;
    };
    LineTw<LOGL, PRE> W;
    if (!a.zero) W.load(tw, t);
    if (!early) wait();
    float2 x[8];
    if (PRE) {
        float2 u[8], E[8], hv[DIM - 1][8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            u[k] = a.uj ? pair(a.uj, bo, k) : make_float2(0.f, 0.f);
            x[k] = u[k];
            if (a.stage == 2) x[k] = pair(us, bo, k);
            E[k] = csub(x[k], u[k]);
        }
        if (a.u_out) {
            if (a.src_in) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 s = pair(a.src_in, bo, k);
                    E[k] = make_float2(fmaf(a.h, s.x, E[k].x), fmaf(a.h, s.y, E[k].y));
                }
            } else if (a.gm) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 s = source(k);
                    if (a.src_out) put(a.src_out, 0, k, s);
                    E[k] = make_float2(fmaf(a.h, s.x, E[k].x), fmaf(a.h, s.y, E[k].y));
                }
            }
#pragma unroll
            for (int d = 0; d < DIM - 1; ++d)
#pragma unroll
                for (int k = 0; k < 8; ++k) hv[d][k] = cscale(pair(a.v, d * N, k), -a.h);
        }
        if (!a.zero) {
            row_deriv<LOGL>(x, t, q, sm, W);
            if (a.u_out) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 w = cscale(pair(a.v, (DIM - 1) * N, k), -a.h);
                    E[k] = make_float2(fmaf(w.x, x[k].x, E[k].x), fmaf(w.y, x[k].y, E[k].y));
                }
            }
        }
        if (early) wait();
        float2 D[DIM - 1][8];
#pragma unroll
        for (int d = 0; d < DIM - 1; ++d)
#pragma unroll
            for (int k = 0; k < 8; ++k) D[d][k] = a.zero ? make_float2(0.f, 0.f) : pair(a.D[d], bo, k);
        if (a.grad_out) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
#pragma unroll
                for (int d = 0; d < DIM - 1; ++d) put(a.grad_out, go + d * N, k, D[d][k]);
                put(a.grad_out, go + (DIM - 1) * N, k, a.zero ? make_float2(0.f, 0.f) : x[k]);
            }
        }
        if (a.u_out) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
#pragma unroll
                for (int d = 0; d < DIM - 1; ++d)
                    E[k] = make_float2(fmaf(hv[d][k].x, D[d][k].x, E[k].x), fmaf(hv[d][k].y, D[d][k].y, E[k].y));
                put(a.u_out, bo, k, make_float2(fmaf(c, E[k].x, u[k].x), fmaf(c, E[k].y, u[k].y)));
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = a.zero ? make_float2(0.f, 0.f) : pair(us, bo, k);
        if (!a.zero) row_deriv<LOGL>(x, t, q, sm, W);
#pragma unroll
        for (int k0 = 0; k0 < 8; k0 += BATCH) {
            float2 u[BATCH], E[BATCH], D[DIM - 1][BATCH];
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int k = k0 + i;
#pragma unroll
                for (int d = 0; d < DIM - 1; ++d) D[d][i] = a.zero ? make_float2(0.f, 0.f) : pair(a.D[d], bo, k);
                if (a.u_out) {
                    u[i] = a.uj ? pair(a.uj, bo, k) : make_float2(0.f, 0.f);
                    E[i] = a.stage == 2 ? csub(pair(a.us, bo, k), u[i]) : make_float2(0.f, 0.f);
                    if (a.src_in || a.gm) {
                        const float2 s = a.src_in ? pair(a.src_in, bo, k) : source(k);
                        if (a.src_out) put(a.src_out, 0, k, s);
                        E[i] = make_float2(fmaf(a.h, s.x, E[i].x), fmaf(a.h, s.y, E[i].y));
                    }
                    if (!a.zero) {
                        const float2 w = cscale(pair(a.v, (DIM - 1) * N, k), -a.h);
                        E[i] = make_float2(fmaf(w.x, x[k].x, E[i].x), fmaf(w.y, x[k].y, E[i].y));
#pragma unroll
                        for (int d = 0; d < DIM - 1; ++d) {
                            const float2 y = cscale(pair(a.v, d * N, k), -a.h);
                            E[i] = make_float2(fmaf(y.x, D[d][i].x, E[i].x), fmaf(y.y, D[d][i].y, E[i].y));
                        }
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int k = k0 + i;
                if (a.grad_out) {
#pragma unroll
                    for (int d = 0; d < DIM - 1; ++d) put(a.grad_out, go + d * N, k, D[d][i]);
                    put(a.grad_out, go + (DIM - 1) * N, k, x[k]);
                }
                if (a.u_out) put(a.u_out, bo, k, make_float2(fmaf(c, E[i].x, u[i].x), fmaf(c, E[i].y, u[i].y)));
            }
        }
    }
}

template <int LOGL, int DIM, bool PRE, bool FULL, int BATCH, class Wait>
__device__ __forceinline__ void adj_row_body(const AdjStage<DIM>& a, uint32_t N, int lines, float2* sm,
                                             const float2* __restrict__ tw, Wait wait) {
    constexpr int L = 1 << LOGL, T = L >> 3;
    const int q = threadIdx.x / T, t = threadIdx.x - q * T;
    const uint32_t r0 = (blockIdx.x * lines + q) * 2 * L + t, r1 = r0 + L;
    const float c = a.stage == 2 ? 0.5f : 1.f;
    auto pair = [&](const float* p, uint32_t o, int k) { return make_float2(p[o + r0 + k * T], p[o + r1 + k * T]); };
    auto put = [&](float* p, uint32_t o, int k, float2 w) { p[o + r0 + k * T] = w.x; p[o + r1 + k * T] = w.y; };
    LineTw<LOGL, PRE> W;
    W.load(tw, t);
    if (!PRE) wait();
    float2 x[8], u[8], E[PRE ? 8 : 1];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float2 s;
        if (PRE) {
            u[k] = pair(a.lj, 0, k);
            s = a.stage == 2 ? pair(a.ls, 0, k) : u[k];
            E[PRE ? k : 0] = csub(s, u[k]);
        } else {
            s = pair(a.stage == 2 ? a.ls : a.lj, 0, k);
        }
        const float2 w = pair(a.v, (DIM - 1) * N, k);
        x[k] = make_float2(__fmul_rn(s.x, w.x), __fmul_rn(s.y, w.y));
        if (FULL) {
            const float2 l = pair(a.lsrc, 0, k), m = pair(a.vt, (DIM - 1) * N, k);
            x[k] = make_float2(fmaf(l.x, m.x, x[k].x), fmaf(l.y, m.y, x[k].y));
        }
    }
    // 2-D: the gradient history comes from HBM on large grids, so it is fetched ahead of the wait as
    // well (3-D blocks are held to 128 registers and live on warps in flight instead)
    constexpr bool EARLYB = PRE && !FULL && DIM == 2;
    float2 gE[EARLYB ? DIM : 1][8], bE[EARLYB ? DIM : 1][8];
    if (EARLYB && a.b) {
#pragma unroll
        for (int d = 0; d < (EARLYB ? DIM : 0); ++d)
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                gE[d][k] = pair(a.gm, d * N, k);
                bE[d][k] = pair(a.b, d * N, k);
            }
    }
    row_deriv<LOGL>(x, t, q, sm, W);
    if (PRE) wait();
    constexpr int B = PRE ? 8 : BATCH;
#pragma unroll
    for (int k0 = 0; k0 < 8; k0 += B) {
        float2 D[DIM - 1][B], gb[DIM][B], bb[DIM][B];
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int k = k0 + i;
#pragma unroll
            for (int d = 0; d < DIM - 1; ++d) D[d][i] = pair(a.D[d], 0, k);
            if (a.b && !PRE) {
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    gb[d][i] = pair(a.gm, d * N, k);
                    bb[d][i] = pair(a.b, d * N, k);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int k = k0 + i;
            float2 dv = x[k], e;
            if (PRE) {
                e = E[PRE ? k : 0];
            } else {
                u[k] = pair(a.lj, 0, k);
                e = a.stage == 2 ? csub(pair(a.ls, 0, k), u[k]) : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int d = 0; d < DIM - 1; ++d) dv = cadd(dv, D[d][i]);
            u[k].x = fmaf(c, fmaf(a.h, dv.x, e.x), u[k].x);
            u[k].y = fmaf(c, fmaf(a.h, dv.y, e.y), u[k].y);
        }
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int k = k0 + i;
            put(a.l_out, 0, k, u[k]);
            if (a.b && !PRE) {
                const float2 l = cscale(u[k], a.w);
                float2 m = make_float2(0.f, 0.f);
                if (FULL) m = cscale(pair(a.lsrc, 0, k), a.w);
#pragma unroll
                for (int d = 0; d < DIM; ++d) {
                    float2 w = make_float2(fmaf(l.x, gb[d][i].x, bb[d][i].x), fmaf(l.y, gb[d][i].y, bb[d][i].y));
                    if (FULL) {
                        const float2 g = pair(a.gmt, d * N, k);
                        w = make_float2(fmaf(m.x, g.x, w.x), fmaf(m.y, g.y, w.y));
                    }
                    put(a.b, d * N, k, w);
                }
            }
        }
    }
    if (!PRE || !a.b) return;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        float2 b[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float2 g = EARLYB ? gE[EARLYB ? d : 0][k] : pair(a.gm, d * N, k);
            const float2 o = EARLYB ? bE[EARLYB ? d : 0][k] : pair(a.b, d * N, k), l = cscale(u[k], a.w);
            b[k] = make_float2(fmaf(l.x, g.x, o.x), fmaf(l.y, g.y, o.y));
            if (FULL) {
                const float2 m = cscale(pair(a.lsrc, 0, k), a.w), gt = pair(a.gmt, d * N, k);
                b[k] = make_float2(fmaf(m.x, gt.x, b[k].x), fmaf(m.y, gt.y, b[k].y));
            }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) put(a.b, d * N, k, b[k]);
    }
}

// ---- deformation gradient (Eq. (e:def-grad)), 2-D ----
// Heun stage of d_t F + (v . grad) F = (grad v) F.  blockIdx.y is the column b of F: F_0b and F_1b
// of one row travel as one complex line, so a thread holds both entries the product couples.
// F planes (F11, F12, F21, F22); D their x^1 derivatives; gv planes (d1 v1, d2 v1, d1 v2, d2 v2).
// As in adv_row_body the row transform and everything that does not need D precede the wait.
struct DefGradStage {
    const float* D;
    const float* F;
    const float* Fs;   // stage 2: F*
    const float* v;
    const float* gv;
    float* out;
    float h;
    int stage;
};

template <int LOGL, class Wait>
__device__ __forceinline__ void defgrad_row_body(const DefGradStage& a, uint32_t N, int lines, float2* sm,
                                                 const float2* __restrict__ tw, Wait wait) {
    constexpr int L = 1 << LOGL, T = L >> 3;
    const int q = threadIdx.x / T, t = threadIdx.x - q * T;
    const uint32_t r = (blockIdx.x * lines + q) * L + t;
    const uint32_t p0 = blockIdx.y * N, p1 = (2 + blockIdx.y) * N;
    const float c = a.stage == 2 ? 0.5f : 1.f;
    LineTw<LOGL, true> W;
    W.load(tw, t);
    float2 x[8], u[8], E[8], w1[8];
    const float* Fs = a.stage == 2 ? a.Fs : a.F;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t i = r + k * T;
        x[k] = make_float2(Fs[p0 + i], Fs[p1 + i]);
        u[k] = a.stage == 2 ? make_float2(a.F[p0 + i], a.F[p1 + i]) : x[k];
        const float g00 = a.gv[i], g01 = a.gv[N + i], g10 = a.gv[2 * N + i], g11 = a.gv[3 * N + i];
        E[k] = csub(x[k], u[k]);
        E[k].x = fmaf(a.h, fmaf(g00, x[k].x, __fmul_rn(g01, x[k].y)), E[k].x);
        E[k].y = fmaf(a.h, fmaf(g10, x[k].x, __fmul_rn(g11, x[k].y)), E[k].y);
        w1[k].x = -a.h * a.v[i];
        w1[k].y = -a.h * a.v[N + i];
    }
    row_deriv<LOGL>(x, t, q, sm, W);
#pragma unroll
    for (int k = 0; k < 8; ++k) E[k] = make_float2(fmaf(w1[k].y, x[k].x, E[k].x), fmaf(w1[k].y, x[k].y, E[k].y));
    wait();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t i = r + k * T;
        x[k] = make_float2(a.D[p0 + i], a.D[p1 + i]);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t i = r + k * T;
        E[k] = make_float2(fmaf(w1[k].x, x[k].x, E[k].x), fmaf(w1[k].x, x[k].y, E[k].y));
        a.out[p0 + i] = fmaf(c, E[k].x, u[k].x);
        a.out[p1 + i] = fmaf(c, E[k].y, u[k].y);
    }
}

// out = d/dx of f along the contiguous axis (+ add, nullable: read after the wait) for pairs
// [tile lines, (tile + 1) lines) of npairs row pairs
template <int LOGL, bool EARLY, class Wait>
__device__ __forceinline__ void drow_body(const float* f, const float* add, float* out, int tile, int lines, int npairs,
                                          float2* sm, const float2* __restrict__ tw, Wait wait) {
    constexpr int L = 1 << LOGL, T = L >> 3;
    const int q = threadIdx.x / T, t = threadIdx.x - q * T;
    const int pr = tile * lines + q;
    const bool on = pr < npairs;
    const uint32_t r0 = (uint32_t)pr * 2 * L + t, r1 = r0 + L;
    LineTw<LOGL, true> W;
    W.load(tw, t);
    if (!EARLY) wait();
    float2 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = on ? make_float2(f[r0 + k * T], f[r1 + k * T]) : make_float2(0.f, 0.f);
    row_deriv<LOGL>(x, t, q, sm, W);
    if (EARLY) wait();
    if (!on) return;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (add) x[k] = cadd(x[k], make_float2(add[r0 + k * T], add[r1 + k * T]));
        out[r0 + k * T] = x[k].x;
        out[r1 + k * T] = x[k].y;
    }
}
