// Three-dimensional registration operators on the GPU: the reduced gradient and the
// Gauss-Newton Hessian matvec of the H1-regularized problem on an n1 x n2 x n3 periodic
// box (the paper's equations of Sec. 3 for d = 3: state Eq. (e:state-eq-elim), adjoint
// Eq. (e:adj-eq-elim), incremental state and adjoint Eqs. (e:inc-state-eq-elim),
// (e:inc-adj-eq-elim), body forces and the projection K of Eq. (e:project-body-force)),
// with the same discretization as the 2-D path: Heun's RK2 in pseudo-time, trapezoidal
// time quadrature, pseudospectral derivatives with odd symbols k~ (Nyquist entry zero)
// and the full even symbol |k|^2.
//
// Layout: real fields are n1 x n2 x n3 floats, index (i1 n2 + i2) n3 + i3; vector fields
// three such fields back to back.
//
// Transport solves: a spectral derivative along one axis needs the transform of that axis
// only (deriv.cuh), so a Heun stage is two launches and no three-dimensional transform:
// k3_d12 takes the derivatives along axes 1 and 2 (the two as different blocks of one
// launch), k3_adv / k3_adj take the one along axis 3 and update.
// Assembly (regularization and projection, which couple the axes): half spectra along axis 3,
// n1 x n2 x (n3 / 2 + 1) complex entries per field, in five launches: rows real to complex,
// axis 2, axis 1 forward with the multiplier and back, axis 2 back, rows complex to real.
//
// 128^3, nt = 16 matvec: 42.5 ms with full complex 3-D transforms in every stage, 1.54 ms now; about
// 10 us a stage in k3_d12 (shared memory and FP32 issue) and 12 us in the row kernels (L2 and, for
// the gradient history, HBM: 4 TB/s).  64 x 128 x 32, nt = 5 gradient: 4.62 -> 0.27 ms.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <string>
#include <utility>
#include <vector>

#include "deriv.cuh"
#include "internal.h"
#include "launch.cuh"

namespace {

constexpr int R3_THREADS = 256;
constexpr int R3_BLOCKS = 608;  // 4 per SM of a GB300 for the grid-stride kernels

struct Dims3 {
    int n1, n2, n3;
    long long N;
    int l1, l2, l3;  // log2
    int W1;          // n3 / 2 + 1: entries of a half-spectrum row
    long long NS;    // n1 n2 W1
};

#define DISPATCH3(LOG, ...)                                   \
    switch (LOG) {                                            \
        case 3: { constexpr int LG = 3; __VA_ARGS__; } break; \
        case 4: { constexpr int LG = 4; __VA_ARGS__; } break; \
        case 5: { constexpr int LG = 5; __VA_ARGS__; } break; \
        case 6: { constexpr int LG = 6; __VA_ARGS__; } break; \
        case 7: { constexpr int LG = 7; __VA_ARGS__; } break; \
        case 8: { constexpr int LG = 8; __VA_ARGS__; } break; \
        default: break;                                       \
    }

#define GRID_STRIDE(i, n) for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (n); i += (long long)gridDim.x * blockDim.x)

// ---- transport ----
// derivatives along axes 1 (blocks [0, tiles1)) and 2 (the rest): columns of float2 (deriv.cuh)
struct D12Args {
    DColArgs a1, a2;
    ColMap m1, m2;
    int log1, log2, tiles1;
};
template <int LOGL, bool WIDE>
__device__ __forceinline__ void d12_role(const DColArgs& a, const ColMap& m, int tile, float2* sm, const float2* __restrict__ tw) {
    if constexpr (WIDE && LOGL >= 7) dcol_wide_body<LOGL>(a, m, tile, sm, tw, pdl_entry);
    else dcol_body<LOGL, 10 - LOGL, true>(a, m, tile, sm, tw, pdl_entry);
}
template <bool WIDE>
__global__ void __launch_bounds__(128, 4) k3_d12(D12Args a, const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    if ((int)blockIdx.x < a.tiles1) {
        DISPATCH3(a.log1, d12_role<LG, WIDE>(a.a1, a.m1, blockIdx.x, sm, tw));
    } else {
        DISPATCH3(a.log2, d12_role<LG, WIDE>(a.a2, a.m2, blockIdx.x - a.tiles1, sm, tw));
    }
}

template <int LOGL>
__global__ void __launch_bounds__(128, 4) k3_adv(AdvStage<3> a, long long N, int lines, const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    adv_row_body<LOGL, 3, true, 8>(a, (uint32_t)N, lines, sm, tw, pdl_entry);
}

template <int LOGL>
__global__ void __launch_bounds__(128, 4) k3_adj(AdjStage<3> a, long long N, int lines, const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    adj_row_body<LOGL, 3, true, false, 8>(a, (uint32_t)N, lines, sm, tw, pdl_entry);
}

// lam(1) = ca a + cb c (a nullable) and b = w lam grad m(1): the start of an adjoint solve
__global__ void __launch_bounds__(R3_THREADS) k3_adj_init(const float* __restrict__ a, float ca,
                                                          const float* __restrict__ c, float cb, float* lam, float* b,
                                                          const float* __restrict__ gm, float w, long long N) {
    pdl_entry();
    GRID_STRIDE(i, N) {
        float l = cb * c[i];
        if (a) l = fmaf(ca, a[i], l);
        lam[i] = l;
#pragma unroll
        for (int d = 0; d < 3; ++d) b[d * N + i] = w * l * gm[d * N + i];
    }
}

// ---- assembly: half spectra ----
// rows of up to six real fields (0..2 from p0, 3..5 from p1, planes of N) to half spectra along
// axis 3: two rows per complex transform, split into entries 0..n3/2 of each
template <int LOGL>
__global__ void __launch_bounds__(128) k3_r2c(const float* __restrict__ p0, const float* __restrict__ p1, float2* S,
                                              Dims3 D, int lines, const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    constexpr int L = 1 << LOGL, T = L >> 3, H = L >> 1;
    const int q = threadIdx.x / T, t = threadIdx.x - q * T;
    const int f = blockIdx.y;
    const float* src = (f < 3 ? p0 + f * D.N : p1 + (f - 3) * D.N);
    const long long row = ((long long)blockIdx.x * lines + q) * 2;
    LineTw<LOGL, false> W;
    W.load(tw, t);
    pdl_entry();
    float2 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = make_float2(src[row * L + t + k * T], src[(row + 1) * L + t + k * T]);
    float2* cur = sm + 2 * q * fft_buf(L);
    float2* nxt = cur + fft_buf(L);
    line_fft<LOGL, false, 1>(x, t, cur, nxt, RowSync<LOGL>(), W);
#pragma unroll
    for (int k = 0; k < 8; ++k) nxt[fft_pad(t + k * T)] = x[k];
    RowSync<LOGL>()();
    float2* o0 = S + f * D.NS + row * D.W1;
    float2* o1 = o0 + D.W1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int e = t + k * T;
        const float2 z = x[k], y = nxt[fft_pad((L - e) & (L - 1))];
        o0[e] = make_float2(0.5f * (z.x + y.x), 0.5f * (z.y - y.y));
        o1[e] = make_float2(0.5f * (z.y + y.y), -0.5f * (z.x - y.x));
    }
    if (t == 0) {
        const float2 z = x[4];  // entry H = 4 T
        o0[H] = make_float2(z.x, 0.f);
        o1[H] = make_float2(z.y, 0.f);
    }
}

// the inverse of k3_r2c for the three planes of out (the 1 / N is in the multiplier)
template <int LOGL>
__global__ void __launch_bounds__(128) k3_c2r(const float2* __restrict__ S, float* out, Dims3 D, int lines,
                                              const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    constexpr int L = 1 << LOGL, T = L >> 3, H = L >> 1;
    const int q = threadIdx.x / T, t = threadIdx.x - q * T;
    const int f = blockIdx.y;
    const long long row = ((long long)blockIdx.x * lines + q) * 2;
    LineTw<LOGL, false> W;
    W.load(tw, t);
    pdl_entry();
    const float2* s0 = S + f * D.NS + row * D.W1;
    const float2* s1 = s0 + D.W1;
    float2 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int p = t + k * T;
        const int e = p <= H ? p : L - p;
        const float2 A = s0[e], B = s1[e];
        if (p == 0 || p == H) x[k] = make_float2(A.x, B.x);
        else x[k] = p < H ? make_float2(A.x - B.y, A.y + B.x) : make_float2(A.x + B.y, -A.y + B.x);
    }
    float2* cur = sm + 2 * q * fft_buf(L);
    float2* nxt = cur + fft_buf(L);
    line_fft<LOGL, true, 1>(x, t, cur, nxt, RowSync<LOGL>(), W);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        out[f * D.N + row * L + t + k * T] = x[k].x;
        out[f * D.N + (row + 1) * L + t + k * T] = x[k].y;
    }
}

// axis 2 of nf half spectra in place: column l = ((f n1 + i1) W1 + e), entries W1 apart
template <int LOGL, bool INV>
__global__ void __launch_bounds__(128) k3_axis2(float2* S, Dims3 D, int ncols, const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    constexpr int L = 1 << LOGL, T = L >> 3, C = 1024 / L;
    const int c = threadIdx.x & (C - 1), t = threadIdx.x / C;
    const int l = blockIdx.x * C + c;
    const bool on = l < ncols;
    const int g = l / D.W1;
    float2* p = S + ((long long)g * D.n2) * D.W1 + (l - g * D.W1);
    LineTw<LOGL, false> W;
    W.load(tw, t);
    pdl_entry();
    float2 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = on ? p[(long long)(t + k * T) * D.W1] : make_float2(0.f, 0.f);
    float2* cur = sm + C * fft_buf(L) + c;
    float2* nxt = sm + c;
    line_fft<LOGL, INV, C>(x, t, cur, nxt, [] { __syncthreads(); }, W);
    if (on) {
#pragma unroll
        for (int k = 0; k < 8; ++k) p[(long long)(t + k * T) * D.W1] = x[k];
    }
}

enum { A3_ASSEMBLE = 0, A3_PRECOND = 1, A3_ENERGY = 2 };
struct Axis1Args {
    const float2* B;   // three spectra (A3_ASSEMBLE: of b; A3_PRECOND: of r; A3_ENERGY: unused)
    const float2* V;   // three spectra of v (A3_ASSEMBLE, A3_ENERGY)
    float2* out;       // three spectra
    double* part;      // nullable: per-block energy sums (reg, w), 3 doubles per block (the first 0)
    float beta, beta_w, invN;
    int mode;          // K^: 0 identity, 1 incompressible, 2 mass source
};

__device__ __forceinline__ float k_odd(int i, int n) { return i < n / 2 ? (float)i : (i == n / 2 ? 0.f : (float)(i - n)); }
__device__ __forceinline__ float k_even(int i, int n) { return i < n / 2 ? (float)i : (float)(i - n); }

// fixed-order sum over the block (a power of two of threads, at most 256)
__device__ __forceinline__ double block_sum3(double v) {
    __shared__ double sh[R3_THREADS];
    __syncthreads();
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    return sh[0];
}

// axis 1: forward, multiplier, inverse.  Column l = i2 W1 + e, entries n2 W1 apart.
//   A3_ASSEMBLE: beta |k|^2 V + K^ B, K^ = I - k~ k~^T / (|k~|^2 [+ beta |k|^2 / (beta_w (1 + |k|^2))])
//   A3_PRECOND:  B / (beta |k|^2), the k = 0 symbol of A replaced by 1 (App. E)
//   A3_ENERGY:   no output; sums of |k|^2 |V|^2 and (1 + |k|^2) |k~ . V|^2 over the full spectrum
//                (an entry with 0 < e < n3 / 2 stands for itself and its conjugate)
template <int LOGL, int OP>
__global__ void __launch_bounds__(128) k3_axis1(Axis1Args a, Dims3 D, int ncols, const float2* __restrict__ tw) {
    extern __shared__ __align__(16) float2 sm[];
    constexpr int L = 1 << LOGL, T = L >> 3, C = 1024 / L;
    constexpr int NV = OP == A3_PRECOND ? 0 : 3, NB = OP == A3_ENERGY ? 0 : 3;
    const int c = threadIdx.x & (C - 1), t = threadIdx.x / C;
    const int l = blockIdx.x * C + c;
    const bool on = l < ncols;
    const long long S = (long long)D.n2 * D.W1;
    LineTw<LOGL, false> W;
    W.load(tw, t);
    pdl_entry();
    float2* cur = sm + C * fft_buf(L) + c;
    float2* nxt = sm + c;
    auto sync = [] { __syncthreads(); };
    float2 xv[NV > 0 ? 3 : 1][8], xb[NB > 0 ? 3 : 1][8];
#pragma unroll
    for (int d = 0; d < NV; ++d) {
#pragma unroll
        for (int k = 0; k < 8; ++k) xv[d][k] = on ? a.V[d * D.NS + l + (t + k * T) * S] : make_float2(0.f, 0.f);
        line_fft<LOGL, false, C>(xv[d], t, cur, nxt, sync, W);
    }
#pragma unroll
    for (int d = 0; d < NB; ++d) {
#pragma unroll
        for (int k = 0; k < 8; ++k) xb[d][k] = on ? a.B[d * D.NS + l + (t + k * T) * S] : make_float2(0.f, 0.f);
        line_fft<LOGL, false, C>(xb[d], t, cur, nxt, sync, W);
    }
    const int i2 = l / D.W1, e = l - i2 * D.W1;
    const float k2 = k_odd(i2, D.n2), e2 = k_even(i2, D.n2);
    const float k3 = e == D.n3 / 2 ? 0.f : (float)e, e3 = (float)e;
    const double ew = (e == 0 || e == D.n3 / 2) ? 1.0 : 2.0;
    double er = 0.0, eww = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int p = t + k * T;
        const float k1 = k_odd(p, L), e1 = k_even(p, L);
        const float kk = e1 * e1 + e2 * e2 + e3 * e3;
        const float kd[3] = {k1, k2, k3};
        if (OP != A3_PRECOND && a.part) {
            double s = 0.0, wr = 0.0, wi = 0.0;
#pragma unroll
            for (int d = 0; d < NV; ++d) {
                s += (double)xv[d][k].x * xv[d][k].x + (double)xv[d][k].y * xv[d][k].y;
                wr += (double)kd[d] * xv[d][k].x;
                wi += (double)kd[d] * xv[d][k].y;
            }
            er += ew * (double)kk * s;
            eww += ew * (1.0 + (double)kk) * (wr * wr + wi * wi);
        }
        if (OP == A3_ASSEMBLE) {
            const float ko = k1 * k1 + k2 * k2 + k3 * k3;
            float cre = 0.f, cim = 0.f;
            if (a.mode != 0 && ko > 0.f) {
                const float denom = a.mode == 1 ? ko : ko + a.beta * kk / (a.beta_w * (1.f + kk));
                cre = (k1 * xb[0][k].x + k2 * xb[NB > 1 ? 1 : 0][k].x + k3 * xb[NB > 2 ? 2 : 0][k].x) / denom;
                cim = (k1 * xb[0][k].y + k2 * xb[NB > 1 ? 1 : 0][k].y + k3 * xb[NB > 2 ? 2 : 0][k].y) / denom;
            }
#pragma unroll
            for (int d = 0; d < NB; ++d) {
                const float2 v = xv[d < NV ? d : 0][k];
                const float br = xb[d][k].x - kd[d] * cre, bi = xb[d][k].y - kd[d] * cim;
                xb[d][k] = make_float2((a.beta * kk * v.x + br) * a.invN, (a.beta * kk * v.y + bi) * a.invN);
            }
        } else if (OP == A3_PRECOND) {
            const float s = a.invN / (a.beta * (kk > 0.f ? kk : 1.f));
#pragma unroll
            for (int d = 0; d < NB; ++d) xb[d][k] = make_float2(xb[d][k].x * s, xb[d][k].y * s);
        }
    }
    if (OP != A3_PRECOND && a.part) {
        if (!on) er = eww = 0.0;
        const double s1 = block_sum3(er), s2 = block_sum3(eww);
        if (threadIdx.x == 0) {
            a.part[blockIdx.x * 3] = 0.0;
            a.part[blockIdx.x * 3 + 1] = s1;
            a.part[blockIdx.x * 3 + 2] = s2;
        }
    }
#pragma unroll
    for (int d = 0; d < NB; ++d) {
        line_fft<LOGL, true, C>(xb[d], t, cur, nxt, sync, W);
        if (on) {
#pragma unroll
            for (int k = 0; k < 8; ++k) a.out[d * D.NS + l + (t + k * T) * S] = xb[d][k];
        }
    }
}

// ---- reductions: per-block FP64 partial sums (3 doubles per block), summed in a fixed order by k3_reduce ----
// sum (mR - m1)^2
__global__ void __launch_bounds__(R3_THREADS) k3_data_part(const float* __restrict__ mR, const float* __restrict__ m1,
                                                           long long N, double* part) {
    pdl_entry();
    double a = 0.0;
    GRID_STRIDE(i, N) {
        const double d = (double)mR[i] - (double)m1[i];
        a += d * d;
    }
    const double s = block_sum3(a);
    if (threadIdx.x < 3) part[blockIdx.x * 3 + threadIdx.x] = threadIdx.x == 0 ? s : 0.0;
}

__global__ void __launch_bounds__(R3_THREADS) k3_reduce(const double* __restrict__ part, int nblk, double* out) {
    pdl_entry();
    double a[3] = {0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblk; b += blockDim.x)
#pragma unroll
        for (int q = 0; q < 3; ++q) a[q] += part[b * 3 + q];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double s = block_sum3(a[q]);
        if (threadIdx.x == 0) out[q] = s;
    }
}

// sum_i a_i b_i
__global__ void __launch_bounds__(R3_THREADS) k3_dot_part(const float* __restrict__ a, const float* __restrict__ b,
                                                          long long n, double* part) {
    pdl_entry();
    double t = 0.0;
    GRID_STRIDE(i, n) t += (double)a[i] * (double)b[i];
    const double s = block_sum3(t);
    if (threadIdx.x < 3) part[blockIdx.x * 3 + threadIdx.x] = threadIdx.x == 0 ? s : 0.0;
}

// y = a x + b y (b == 0: y is not read)
__global__ void k3_axpby(const float* x, float* y, long long n, float a, float b) {  // x may be y
    pdl_entry();
    GRID_STRIDE(i, n) y[i] = b != 0.f ? a * x[i] + b * y[i] : a * x[i];
}

}  // namespace

struct reg3_ctx {
    Dims3 D;
    int nt;
    double beta, gamma;
    int kmode;  // 0: K = I (gamma = 0), 1: incompressible (gamma = inf), 2: mass source
    cudaStream_t stream;
    GraphBuild* build;  // launches go into this graph (nullptr: onto `stream`)
    void* slab;  // the allocation behind the device buffers
    float *mT, *mR, *v, *vt, *gm, *y, *ys, *lam, *src, *D1, *D2, *bt;
    float2* S;   // six half spectra: 0..2 of b (and the results), 3..5 of v
    float2* tw;
    double *d_part, *d_sum, *h_sum;
    int npart;   // blocks d_part has room for
    cudaGraphExec_t graphs[4];
    bool have_images, have_lin;
};

namespace {

bool pow2_in(int n, int lo, int hi) { return n >= lo && n <= hi && (n & (n - 1)) == 0; }
int ilog2(int n) { int l = 0; while ((1 << l) < n) ++l; return l; }

template <typename... KArgs, typename... Args>
void launch3(reg3_ctx* c, void (*kern)(KArgs...), dim3 grid, int block, size_t smem, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    launch_cfg<KArgs...>(c->build, cfg, kern, static_cast<KArgs>(args)...);
}

// D1 = d_1 (f mul1), D2 = d_2 (f mul2) (no factor where mul is nullptr)
void d12(reg3_ctx* c, const float* f, const float* mul1, const float* mul2) {
    const Dims3& D = c->D;
    D12Args a;
    a.a1 = DColArgs{f, mul1, nullptr, nullptr, c->D1};
    a.a2 = DColArgs{f, mul2, nullptr, nullptr, c->D2};
    const int nc1 = D.n2 * D.n3 / 2, nc2 = D.n1 * D.n3 / 2;
    a.m1 = ColMap{D.l2 + D.l3 - 1, 0, nc1, nc1};
    a.m2 = ColMap{D.l3 - 1, D.n2 * D.n3 / 2, D.n3 / 2, nc2};
    a.log1 = D.l1;
    a.log2 = D.l2;
    // 16 entries a thread on axes of 128 and 256 points where that leaves several blocks per SM.  Matvec,
    // nt = 4, us with 16 / with 8: 256 x 128 x 128 1061 / 1139, 128^3 488 / 524, 256 x 128 x 32 381 / 396,
    // 64 x 128 x 128 263 / 265; below 2^20 points it depends on the box: 128 x 64 x 64 203 / 203,
    // 128 x 128 x 16 192 / 229, 16 x 128 x 256 180 / 178, 128 x 16 x 16 120 / 117
    const bool wide = D.N >= (1 << 20);
    auto cols = [&](int n) { return (wide && n >= 128 ? 2048 : 1024) / n; };  // columns of a block
    auto smem = [&](int n) {
        return wide && n >= 128 ? (n == 128 ? Wide<7>::SMEM : Wide<8>::SMEM) : dcol_smem(1024 / n, n);
    };
    const int C1 = cols(D.n1), C2 = cols(D.n2);
    a.tiles1 = (nc1 + C1 - 1) / C1;
    const int tiles2 = (nc2 + C2 - 1) / C2;
    const size_t sh = smem(D.n1) > smem(D.n2) ? smem(D.n1) : smem(D.n2);
    launch3(c, wide ? k3_d12<true> : k3_d12<false>, a.tiles1 + tiles2, 128, sh, a, c->tw);
}

// row kernels: 128 threads a block (64 for small boxes), at most the box's pairs of rows.  Matvec,
// nt = 4, us with 128 / with 64 threads: 32^3 111 / 100, 128 x 32 x 32 140 / 133, 64 x 64 x 32 139 / 128;
// from 2^18 points on the same but for 64^3 149 / 142 and, the reason for the line, 128 x 128 x 16 229 / 291
struct Row3 { int lines, threads, grid; size_t smem; };
Row3 row3(const Dims3& D) {
    Row3 r;
    const int T = D.n3 / 8, pairs = D.n1 * D.n2 / 2;
    const int th = D.N >= (1 << 18) ? 128 : 64;
    r.lines = th / T;
    if (r.lines > pairs) r.lines = pairs;
    r.threads = r.lines * T;
    r.grid = pairs / r.lines;
    r.smem = drow_smem(r.lines, D.n3);
    return r;
}

void adv(reg3_ctx* c, const AdvStage<3>& a) {
    const Row3 r = row3(c->D);
    DISPATCH3(c->D.l3, launch3(c, k3_adv<LG>, r.grid, r.threads, r.smem, a, c->D.N, r.lines, c->tw));
}
void adj(reg3_ctx* c, const AdjStage<3>& a) {
    const Row3 r = row3(c->D);
    DISPATCH3(c->D.l3, launch3(c, k3_adj<LG>, r.grid, r.threads, r.smem, a, c->D.N, r.lines, c->tw));
}

// state (vt == nullptr: y from mT into c->y, gradient history into c->gm) or incremental state
// (source grad m_j . vt from the stored history, from 0, into c->y)
void forward_solve(reg3_ctx* c, const float* vt) {
    const long long N = c->D.N;
    const float h = 1.f / c->nt;
    float* y = c->y;
    AdvStage<3> a = {};
    a.D[0] = c->D1;
    a.D[1] = c->D2;
    a.v = c->v;
    a.vt = vt;
    a.h = h;
    for (int j = 0; j < c->nt; ++j) {
        const float* yj = j > 0 ? y : (vt ? nullptr : c->mT);
        a.uj = yj;
        a.us = nullptr;
        a.stage = 1;
        a.u_out = c->ys;
        a.zero = yj ? 0 : 1;
        a.late = a.zero;  // the first launch of the solve
        a.src_in = (vt && j > 0) ? c->src : nullptr;
        a.gm = vt ? c->gm + 3 * N * j : nullptr;
        a.src_out = nullptr;
        a.grad_out = vt ? nullptr : c->gm + 3 * N * j;
        if (yj) d12(c, yj, nullptr, nullptr);
        adv(c, a);
        d12(c, c->ys, nullptr, nullptr);
        a.us = c->ys;
        a.stage = 2;
        a.u_out = y;
        a.zero = a.late = 0;
        a.src_in = nullptr;
        a.gm = vt ? c->gm + 3 * N * (j + 1) : nullptr;
        a.src_out = (vt && j + 1 < c->nt) ? c->src : nullptr;
        a.grad_out = nullptr;
        adv(c, a);
    }
    if (!vt) {  // grad m(t = 1) completes the history
        d12(c, y, nullptr, nullptr);
        a.uj = y;
        a.us = nullptr;
        a.stage = 1;
        a.u_out = nullptr;
        a.grad_out = c->gm + 3 * N * c->nt;
        adv(c, a);
    }
}

// adjoint transport backward from lam(1) = ca x + cb c->y (x nullable), accumulating out = int lam grad m dt
void adjoint_solve(reg3_ctx* c, const float* x, float ca, float cb, float* out) {
    const long long N = c->D.N;
    const int nt = c->nt;
    const float h = 1.f / nt;
    launch3(c, k3_adj_init, R3_BLOCKS, R3_THREADS, 0, x, ca, c->y, cb, c->lam, out, c->gm + 3 * N * nt, 0.5f * h, N);
    AdjStage<3> a = {};
    a.D[0] = c->D1;
    a.D[1] = c->D2;
    a.v = c->v;
    a.h = h;
    a.lj = c->lam;
    for (int j = nt; j >= 1; --j) {
        d12(c, c->lam, c->v, c->v + N);
        a.stage = 1;
        a.ls = nullptr;
        a.l_out = c->ys;
        a.b = nullptr;
        adj(c, a);
        d12(c, c->ys, c->v, c->v + N);
        a.stage = 2;
        a.ls = c->ys;
        a.l_out = c->lam;
        a.b = out;
        a.gm = c->gm + 3 * N * (j - 1);
        a.w = j == 1 ? 0.5f * h : h;
        adj(c, a);
    }
}

// ---- spectral assembly ----
void rows_r2c(reg3_ctx* c, const float* p0, const float* p1, float2* S, int nf) {
    const Row3 r = row3(c->D);
    DISPATCH3(c->D.l3, launch3(c, k3_r2c<LG>, dim3(r.grid, nf), r.threads, r.smem, p0, p1, S, c->D, r.lines, c->tw));
}
void rows_c2r(reg3_ctx* c, const float2* S, float* out) {
    const Row3 r = row3(c->D);
    DISPATCH3(c->D.l3, launch3(c, k3_c2r<LG>, dim3(r.grid, 3), r.threads, r.smem, S, out, c->D, r.lines, c->tw));
}
// complex column kernels: 128 threads a block
struct Col3 { int grid; size_t smem; };
Col3 col3(int logl, int ncols) {
    const int C = 1024 >> logl;
    return Col3{(ncols + C - 1) / C, dcol_smem(C, 1 << logl)};
}
void axis2(reg3_ctx* c, float2* S, int nf, bool inv) {
    const int nc = nf * c->D.n1 * c->D.W1;
    const Col3 k = col3(c->D.l2, nc);
    if (inv) DISPATCH3(c->D.l2, launch3(c, k3_axis2<LG, true>, k.grid, 128, k.smem, S, c->D, nc, c->tw))
    else DISPATCH3(c->D.l2, launch3(c, k3_axis2<LG, false>, k.grid, 128, k.smem, S, c->D, nc, c->tw))
}
// returns the number of blocks (partial sums, where a.part is set)
int axis1(reg3_ctx* c, int op, double* part) {
    Axis1Args a;
    a.B = c->S;
    a.V = c->S + 3 * c->D.NS;
    a.out = c->S;
    a.part = part;
    a.beta = (float)c->beta;
    a.beta_w = (float)c->gamma;
    a.invN = 1.f / (float)c->D.N;
    a.mode = c->kmode;
    const int nc = c->D.n2 * c->D.W1;
    const Col3 k = col3(c->D.l1, nc);
    if (op == A3_ASSEMBLE)
        DISPATCH3(c->D.l1, launch3(c, k3_axis1<LG, A3_ASSEMBLE>, k.grid, 128, k.smem, a, c->D, nc, c->tw))
    else if (op == A3_PRECOND)
        DISPATCH3(c->D.l1, launch3(c, k3_axis1<LG, A3_PRECOND>, k.grid, 128, k.smem, a, c->D, nc, c->tw))
    else
        DISPATCH3(c->D.l1, launch3(c, k3_axis1<LG, A3_ENERGY>, k.grid, 128, k.smem, a, c->D, nc, c->tw))
    return k.grid;
}

// the parts of J into d_sum: sum (mR - m(1))^2 from the fields, the energies from nblk partial sums
// that follow the data blocks
void reduce_objective(reg3_ctx* c, int nblk) {
    launch3(c, k3_data_part, R3_BLOCKS, R3_THREADS, 0, c->mR, c->y, c->D.N, c->d_part);
    launch3(c, k3_reduce, 1, R3_THREADS, 0, c->d_part, R3_BLOCKS + nblk, c->d_sum);
}

// spectra of beta A x + K b left in c->S (rows_c2r finishes); energy: with the sums of J
void assemble(reg3_ctx* c, const float* x, const float* b, bool energy) {
    rows_r2c(c, b, x, c->S, 6);
    axis2(c, c->S, 6, false);
    const int nblk = axis1(c, A3_ASSEMBLE, energy ? c->d_part + 3 * R3_BLOCKS : nullptr);
    axis2(c, c->S, 3, true);
    if (energy) reduce_objective(c, nblk);
}

int r3_err(const char* what) {
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? REG_OK : reg_fail(REG_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// Run a launch sequence that touches the context's own buffers only: built once per context as a
// CUDA graph and replayed on its working stream.  While the caller captures that stream the
// launches go into the caller's graph instead.
enum { G3_GRADIENT = 0, G3_MATVEC = 1, G3_OBJECTIVE = 2 };
template <typename F>
int run3(reg3_ctx* c, int kind, F&& body) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(c->stream, &cs) != cudaSuccess) return r3_err("capture status");
    if (cs != cudaStreamCaptureStatusNone) {
        body();
        return r3_err("launch");
    }
    if (!c->graphs[kind]) {
        const GraphCalls allow;
        GraphBuild b;
        if (cudaGraphCreate(&b.graph, 0) != cudaSuccess) return r3_err("graph");
        c->build = &b;
        body();
        c->build = nullptr;
        cudaError_t e = b.err;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&c->graphs[kind], b.graph, 0);
        cudaGraphDestroy(b.graph);
        if (e != cudaSuccess) {
            c->graphs[kind] = nullptr;
            cudaGetLastError();
            return reg_fail(REG_ERR_CUDA, std::string("graph: ") + cudaGetErrorString(e));
        }
    }
    cudaGraphLaunch(c->graphs[kind], c->stream);
    return r3_err("graph launch");
}

double objective_value(reg3_ctx* c) {
    const double hv = std::pow(2.0 * M_PI, 3) / (double)c->D.N;
    double J = 0.5 * hv * c->h_sum[0] + 0.5 * c->beta * hv / (double)c->D.N * c->h_sum[1];
    if (c->kmode == 2) J += 0.5 * c->gamma * hv / (double)c->D.N * c->h_sum[2];
    return J;
}

}  // namespace

extern "C" void reg3_destroy(reg3_ctx* c) {
    if (!c) return;
    for (cudaGraphExec_t g : c->graphs)
        if (g) cudaGraphExecDestroy(g);
    cudaFree(c->slab);
    cudaFreeHost(c->h_sum);
    delete c;
}

extern "C" int reg3_create(int n1, int n2, int n3, int nt, double beta, double gamma, reg3_ctx** out) {
    if (!out) return reg_fail(REG_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (!pow2_in(n1, 8, 256) || !pow2_in(n2, 8, 256) || !pow2_in(n3, 8, 256))
        return reg_fail(REG_ERR_ARG, "n1, n2, n3 must be powers of two in [8, 256]");
    if (nt < 1 || nt > 1024) return reg_fail(REG_ERR_ARG, "nt must be in [1, 1024]");
    if (!(beta > 0.0) || !std::isfinite(beta)) return reg_fail(REG_ERR_ARG, "beta must be positive and finite");
    if (!(gamma >= 0.0)) return reg_fail(REG_ERR_ARG, "gamma must be >= 0 (INFINITY: incompressible)");
    reg3_ctx* c = new reg3_ctx();
    c->D = Dims3{n1, n2, n3, (long long)n1 * n2 * n3, ilog2(n1), ilog2(n2), ilog2(n3), n3 / 2 + 1,
                 (long long)n1 * n2 * (n3 / 2 + 1)};
    c->nt = nt;
    c->beta = beta;
    c->gamma = gamma;
    c->kmode = gamma == 0.0 ? 0 : (std::isinf(gamma) ? 1 : 2);
    c->stream = 0;
    c->npart = R3_BLOCKS + col3(c->D.l1, n2 * c->D.W1).grid;
    const size_t N = (size_t)c->D.N;
    // one allocation for all buffers
    size_t used = 0;
    std::vector<std::pair<void**, size_t>> parts;
    auto M = [&](void** p, size_t bytes) {
        parts.emplace_back(p, used);
        used += (bytes + 255) & ~(size_t)255;
    };
    M((void**)&c->mT, sizeof(float) * N);
    M((void**)&c->mR, sizeof(float) * N);
    M((void**)&c->v, sizeof(float) * 3 * N);
    M((void**)&c->vt, sizeof(float) * 3 * N);
    M((void**)&c->gm, sizeof(float) * 3 * N * (nt + 1));
    M((void**)&c->y, sizeof(float) * N);
    M((void**)&c->ys, sizeof(float) * N);
    M((void**)&c->lam, sizeof(float) * N);
    M((void**)&c->src, sizeof(float) * N);
    M((void**)&c->D1, sizeof(float) * N);
    M((void**)&c->D2, sizeof(float) * N);
    M((void**)&c->bt, sizeof(float) * 3 * N);
    M((void**)&c->S, sizeof(float2) * 6 * (size_t)c->D.NS);
    M((void**)&c->tw, sizeof(float2) * REG_TW_TOTAL);
    M((void**)&c->d_part, sizeof(double) * 3 * c->npart);
    M((void**)&c->d_sum, sizeof(double) * 3);
    bool ok = cudaMalloc(&c->slab, used) == cudaSuccess;
    if (ok)
        for (auto& q : parts) *q.first = static_cast<char*>(c->slab) + q.second;
    if (ok && cudaMallocHost((void**)&c->h_sum, sizeof(double) * 3) != cudaSuccess) ok = false;
    if (!ok) {
        cudaGetLastError();
        reg3_destroy(c);
        return reg_fail(REG_ERR_NOMEM, "3-D context allocation failed");
    }
    upload_twiddles(c->tw);
    // A copy from pageable memory may return once its data is staged, and a working stream need not be
    // ordered after the legacy stream (cudaStreamNonBlocking): wait until the table is on the device.
    cudaStreamSynchronize(0);
    const int st = r3_err("3-D context set-up");
    if (st != REG_OK) {
        reg3_destroy(c);
        return st;
    }
    *out = c;
    return REG_OK;
}

extern "C" int reg3_set_stream(reg3_ctx* c, void* stream) {
    if (!c) return reg_fail(REG_ERR_ARG, "ctx is NULL");
    c->stream = (cudaStream_t)stream;
    return REG_OK;
}

extern "C" int reg3_set_images(reg3_ctx* c, const float* mT, const float* mR) {
    if (!c || !mT || !mR) return reg_fail(REG_ERR_ARG, "NULL argument");
    cudaMemcpyAsync(c->mT, mT, sizeof(float) * c->D.N, cudaMemcpyDeviceToDevice, c->stream);
    cudaMemcpyAsync(c->mR, mR, sizeof(float) * c->D.N, cudaMemcpyDeviceToDevice, c->stream);
    c->have_images = true;
    c->have_lin = false;
    return r3_err("reg3_set_images");
}

extern "C" int reg3_gradient(reg3_ctx* c, const float* v, float* g, double* J) {
    if (!c || !v || !g) return reg_fail(REG_ERR_ARG, "NULL argument");
    if (!c->have_images) return reg_fail(REG_ERR_STATE, "reg3_set_images first");
    const long long N = c->D.N;
    cudaMemcpyAsync(c->v, v, sizeof(float) * 3 * N, cudaMemcpyDeviceToDevice, c->stream);
    int st = run3(c, G3_GRADIENT, [&] {
        forward_solve(c, nullptr);                   // m, grad m history
        adjoint_solve(c, c->mR, 1.f, -1.f, c->bt);   // lam(1) = mR - m(1), b
        assemble(c, c->v, c->bt, true);              // beta A v + K b, J parts
    });
    if (st != REG_OK) return st;
    rows_c2r(c, c->S, g);
    cudaMemcpyAsync(c->h_sum, c->d_sum, sizeof(double) * 3, cudaMemcpyDeviceToHost, c->stream);
    st = r3_err("reg3_gradient");
    if (st != REG_OK) return st;
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) return r3_err("reg3_gradient");
    const double Jv = objective_value(c);
    if (J) *J = Jv;
    if (!std::isfinite(Jv)) return reg_fail(REG_ERR_NAN, "objective is not finite");
    c->have_lin = true;
    return REG_OK;
}

extern "C" int reg3_hessian_matvec(reg3_ctx* c, const float* vt, float* Hvt) {
    if (!c || !vt || !Hvt) return reg_fail(REG_ERR_ARG, "NULL argument");
    if (!c->have_lin) return reg_fail(REG_ERR_STATE, "reg3_gradient first (it fixes the linearization point)");
    cudaMemcpyAsync(c->vt, vt, sizeof(float) * 3 * c->D.N, cudaMemcpyDeviceToDevice, c->stream);
    const int st = run3(c, G3_MATVEC, [&] {
        forward_solve(c, c->vt);                       // m~(1)
        adjoint_solve(c, nullptr, 0.f, -1.f, c->bt);   // lam~(1) = -m~(1), b~
        assemble(c, c->vt, c->bt, false);
    });
    if (st != REG_OK) return st;
    rows_c2r(c, c->S, Hvt);
    return r3_err("reg3_hessian_matvec");
}

namespace {

// <a, b> on the grid (trapezoidal weight (2 pi)^3 / N) over 3 N values; synchronous
double inner3(reg3_ctx* c, const float* a, const float* b) {
    launch3(c, k3_dot_part, R3_BLOCKS, R3_THREADS, 0, a, b, 3 * c->D.N, c->d_part);
    launch3(c, k3_reduce, 1, R3_THREADS, 0, c->d_part, R3_BLOCKS, c->d_sum);
    cudaMemcpyAsync(c->h_sum, c->d_sum, sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    cudaStreamSynchronize(c->stream);
    return std::pow(2.0 * M_PI, 3) / (double)c->D.N * c->h_sum[0];
}

void axpby3(reg3_ctx* c, const float* x, float* y, float a, float b) {
    launch3(c, k3_axpby, R3_BLOCKS, R3_THREADS, 0, x, y, 3 * c->D.N, a, b);
}

void precond3(reg3_ctx* c, const float* r, float* out) {
    rows_r2c(c, r, nullptr, c->S, 3);
    axis2(c, c->S, 3, false);
    axis1(c, A3_PRECOND, nullptr);
    axis2(c, c->S, 3, true);
    rows_c2r(c, c->S, out);
}

// J at x (one state solve; the gradient history is overwritten, which Algorithm 1 allows:
// the next gradient evaluation rebuilds it at the accepted point)
double objective3(reg3_ctx* c, const float* x) {
    cudaMemcpyAsync(c->v, x, sizeof(float) * 3 * c->D.N, cudaMemcpyDeviceToDevice, c->stream);
    c->have_lin = false;
    const int st = run3(c, G3_OBJECTIVE, [&] {
        forward_solve(c, nullptr);
        rows_r2c(c, c->v, nullptr, c->S + 3 * c->D.NS, 3);
        axis2(c, c->S + 3 * c->D.NS, 3, false);
        reduce_objective(c, axis1(c, A3_ENERGY, c->d_part + 3 * R3_BLOCKS));
    });
    if (st != REG_OK) return NAN;  // the caller's error check reports it
    cudaMemcpyAsync(c->h_sum, c->d_sum, sizeof(double) * 3, cudaMemcpyDeviceToHost, c->stream);
    cudaStreamSynchronize(c->stream);
    return objective_value(c);
}

}  // namespace

extern "C" int reg3_solve(reg3_ctx* c, float* v, double tol, int maxit_newton, int maxit_pcg, double* stats) {
    if (!c || !v) return reg_fail(REG_ERR_ARG, "NULL argument");
    if (!c->have_images) return reg_fail(REG_ERR_STATE, "reg3_set_images first");
    if (!(tol > 0.0) || maxit_newton < 0 || maxit_pcg < 1) return reg_fail(REG_ERR_ARG, "tol > 0, maxit_pcg >= 1");
    const long long N3 = 3 * c->D.N;
    float *g, *vt, *r, *z, *sd, *Hs, *vtrial;
    float** bufs[] = {&g, &vt, &r, &z, &sd, &Hs, &vtrial};
    for (float** b : bufs) *b = nullptr;
    for (float** b : bufs)
        if (cudaMalloc((void**)b, sizeof(float) * N3) != cudaSuccess) {
            cudaGetLastError();
            for (float** q : bufs) cudaFree(*q);
            return reg_fail(REG_ERR_NOMEM, "reg3_solve work vectors");
        }
    int k = 0, nmv = 0, nls = 0, status = REG_OK;
    double J = 0.0, J0 = 0.0, g0 = 0.0, gn = 0.0;
    auto done = [&](int st) {
        if (stats) {
            stats[0] = k;
            stats[1] = nmv;
            stats[2] = nls;
            stats[3] = g0 > 0.0 ? gn / g0 : 0.0;
            stats[4] = J;
            stats[5] = st;
            stats[6] = J0;
        }
        for (float** q : bufs) cudaFree(*q);
        return st;
    };
    const double c1 = 1e-4, rho = 0.5;
    const int max_ls = 20;
    // Algorithm 1 from v = 0: the stopping test is relative to ||g(0)||
    cudaMemsetAsync(v, 0, sizeof(float) * N3, c->stream);
    int st = reg3_gradient(c, v, g, &J);
    if (st != REG_OK) return done(st);
    J0 = J;
    g0 = gn = std::sqrt(inner3(c, g, g));
    while (g0 > 0.0 && gn / g0 > tol) {
        if (k >= maxit_newton) { status = REG_ERR_MAXIT; break; }
        // Algorithm 2: preconditioned CG on H v~ = -g to ||r|| < eta ||g||
        const double eta = std::fmin(0.5, std::sqrt(gn / g0));
        cudaMemsetAsync(vt, 0, sizeof(float) * N3, c->stream);
        axpby3(c, g, r, -1.f, 0.f);  // r = -g
        precond3(c, r, z);
        cudaMemcpyAsync(sd, z, sizeof(float) * N3, cudaMemcpyDeviceToDevice, c->stream);
        double rz = inner3(c, r, z);
        for (int it = 1; it <= maxit_pcg; ++it) {
            st = reg3_hessian_matvec(c, sd, Hs);
            if (st != REG_OK) return done(st);
            ++nmv;
            const double sHs = inner3(c, sd, Hs);
            if (!(sHs > 0.0)) {
                if (it == 1) cudaMemcpyAsync(vt, sd, sizeof(float) * N3, cudaMemcpyDeviceToDevice, c->stream);
                break;
            }
            const float kappa = (float)(rz / sHs);
            axpby3(c, sd, vt, kappa, 1.f);
            axpby3(c, Hs, r, -kappa, 1.f);
            if (std::sqrt(inner3(c, r, r)) < eta * gn) break;
            precond3(c, r, z);
            const double rz_new = inner3(c, z, r);
            axpby3(c, z, sd, 1.f, (float)(rz_new / rz));
            rz = rz_new;
        }
        double gv = inner3(c, g, vt);
        if (gv >= 0.0) {  // not a descent direction: the preconditioned steepest descent step
            precond3(c, g, vt);
            axpby3(c, vt, vt, 0.f, -1.f);
            gv = inner3(c, g, vt);
        }
        // Armijo backtracking on J
        double alpha = 1.0;
        bool accepted = false;
        for (int l = 0; l < max_ls; ++l) {
            cudaMemcpyAsync(vtrial, v, sizeof(float) * N3, cudaMemcpyDeviceToDevice, c->stream);
            axpby3(c, vt, vtrial, (float)alpha, 1.f);
            ++nls;
            // a trial beyond the explicit scheme's stability gives a non-finite J: rejected like any
            // other trial that fails the sufficient-decrease test
            const double Jt = objective3(c, vtrial);
            if (std::isfinite(Jt) && Jt <= J + c1 * alpha * gv) {
                accepted = true;
                break;
            }
            alpha *= rho;
        }
        if (!accepted) { status = REG_ERR_LINESEARCH; break; }
        cudaMemcpyAsync(v, vtrial, sizeof(float) * N3, cudaMemcpyDeviceToDevice, c->stream);
        ++k;
        st = reg3_gradient(c, v, g, &J);
        if (st != REG_OK) return done(st);
        gn = std::sqrt(inner3(c, g, g));
    }
    const int e = r3_err("reg3_solve");
    if (e != REG_OK) return done(e);
    if (status == REG_ERR_LINESEARCH) return done(reg_fail(status, "line search failed"));
    if (status == REG_ERR_MAXIT) return done(reg_fail(status, "Newton iteration cap reached before the tolerance"));
    return done(REG_OK);
}
