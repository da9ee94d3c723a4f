// Launch helpers shared by the 2-D kernel files (kernels.cu, transport.cu): programmatic dependent
// launch, the context's tiles, shared-memory opt-in, dispatch over transform lengths.
#pragma once
#include <cuda_runtime.h>

#include <mutex>
#include <unordered_map>

#include "internal.h"

#define NTHREADS 256
#define NBLK_RED 304  // 2 x 152 SMs

// Programmatic dependent launch: every kernel waits for the grid it depends
// on (it has completed and its writes are visible after the wait) and then
// lets the next kernel in the stream begin launching, so the launch, CTA
// scheduling and prologue of kernel k+1 overlap the tail of kernel k.  Since
// each kernel triggers only after its own wait, a kernel that starts early
// may read, before its wait, anything written two or more launches back
// (the RK2 row-stage kernels prefetch their pointwise operands that way).
// Without a programmatic dependency both instructions are no-ops.
__device__ __forceinline__ void pdl_entry() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launch onto cfg.stream, or as the next node of the graph that is being built: with a programmatic
// edge where the configuration asks for programmatic serialization and the node before is a kernel.
template <typename... KArgs>
static void launch_cfg(GraphBuild* b, const cudaLaunchConfig_t& cfg, void (*kern)(KArgs...), KArgs... args) {
    if (!b) {
        cudaLaunchKernelEx(&cfg, kern, args...);
        return;
    }
    void* params[] = {(void*)&args...};
    cudaKernelNodeParams p = {};
    p.func = (void*)kern;
    p.gridDim = cfg.gridDim;
    p.blockDim = cfg.blockDim;
    p.sharedMemBytes = (unsigned)cfg.dynamicSmemBytes;
    p.kernelParams = params;
    bool early = false;
    for (unsigned i = 0; i < cfg.numAttrs; ++i)
        early = early || (cfg.attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization &&
                          cfg.attrs[i].val.programmaticStreamSerializationAllowed);
    early = early && b->tail_kernel;
    cudaGraphNode_t node = nullptr;
    cudaError_t e = cudaGraphAddKernelNode(&node, b->graph, &b->tail, b->tail && !early ? 1 : 0, &p);
    for (unsigned i = 0; e == cudaSuccess && i < cfg.numAttrs; ++i)
        if (cfg.attrs[i].id == cudaLaunchAttributeClusterDimension)
            e = cudaGraphKernelNodeSetAttribute(node, cudaLaunchAttributeClusterDimension, &cfg.attrs[i].val);
    if (e == cudaSuccess && early) {
        cudaGraphEdgeData edge = {};
        edge.from_port = cudaGraphKernelNodePortProgrammatic;
        edge.type = cudaGraphDependencyTypeProgrammatic;
        e = cudaGraphAddDependencies(b->graph, &b->tail, &node, &edge, 1);
    }
    b->add(e, node, true);
}
// the same for a copy between device buffers
[[maybe_unused]] static void copy_async(GraphBuild* b, cudaStream_t st, void* dst, const void* src, size_t bytes) {
    if (!b) {
        cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, st);
        return;
    }
    cudaGraphNode_t node = nullptr;
    const cudaError_t e = cudaGraphAddMemcpyNode1D(&node, b->graph, &b->tail, b->tail ? 1 : 0, dst, src, bytes,
                                                   cudaMemcpyDeviceToDevice);
    b->add(e, node, false);
}

// Launch with the programmatic-stream-serialization attribute (ctx->pdl) or plainly.
template <typename... KArgs, typename... Args>
static void launch_k(reg_ctx* ctx, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctx->pdl ? 1 : 0;
    launch_cfg<KArgs...>(ctx->build, cfg, kern, static_cast<KArgs>(args)...);
}

[[maybe_unused]] static int rows_per_cta(const reg_ctx* ctx) {
    int R, C, P;
    default_tiles(ctx->n1, ctx->n2, &R, &C, &P);
    return ctx->tileR > 0 ? ctx->tileR : R;
}

[[maybe_unused]] static int cols_per_cta(const reg_ctx* ctx) {
    int R, C, P;
    default_tiles(ctx->n1, ctx->n2, &R, &C, &P);
    return ctx->tileC > 0 ? ctx->tileC : C;
}

// the spectral column kernel's default stays at 64 threads: its row-quad tiles give 64-byte segments
// from two columns on
[[maybe_unused]] static int spec_cols_per_cta(const reg_ctx* ctx) {
    if (ctx->tileR > 0) return ctx->tileC;
    int C = 2;
    while (C * (ctx->n1 / 8) < 64 && C * 2 <= ctx->n2 / 2) C *= 2;
    return C;
}

[[maybe_unused]] static bool prefetch_rows(const reg_ctx* ctx) {
    int R, C, P;
    default_tiles(ctx->n1, ctx->n2, &R, &C, &P);
    return (ctx->tileR > 0 ? ctx->tileP : P) != 0;
}

// Opt in to more than 48 KB of dynamic shared memory once per (device, kernel instantiation)
// and size: the attribute applies to the current device only (contexts on several host
// threads launch concurrently, hence the lock).
struct SmemKey {
    int dev;
    const void* kern;
    bool operator==(const SmemKey& o) const { return dev == o.dev && kern == o.kern; }
};
struct SmemKeyHash {
    size_t operator()(const SmemKey& k) const { return std::hash<const void*>()(k.kern) * 31u + (size_t)k.dev; }
};
template <typename K>
static void set_smem(K kern, size_t bytes) {
    if (bytes <= 32 * 1024) return;  // static shared memory (reductions) also counts toward the 48 KB default
    static std::mutex mu;
    static std::unordered_map<SmemKey, size_t, SmemKeyHash> done;
    int dev = 0;
    cudaGetDevice(&dev);
    const SmemKey key{dev, (const void*)kern};
    std::lock_guard<std::mutex> lock(mu);
    auto it = done.find(key);
    if (it != done.end() && it->second >= bytes) return;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    done[key] = bytes;
}

#define DISPATCH_LOG(LOG, ...)                        \
    switch (LOG) {                                    \
        case 4: { constexpr int LG = 4; __VA_ARGS__; } break;   \
        case 5: { constexpr int LG = 5; __VA_ARGS__; } break;   \
        case 6: { constexpr int LG = 6; __VA_ARGS__; } break;   \
        case 7: { constexpr int LG = 7; __VA_ARGS__; } break;   \
        case 8: { constexpr int LG = 8; __VA_ARGS__; } break;   \
        case 9: { constexpr int LG = 9; __VA_ARGS__; } break;   \
        case 10: { constexpr int LG = 10; __VA_ARGS__; } break; \
        default: break;                               \
    }
