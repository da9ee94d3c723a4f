// Thread-block-cluster primitives and launch set-up shared by the resident transport kernels.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t cl_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// address of this CTA's shared location p in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cl_map(const void* p, int rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ float2 cl_load(uint32_t a) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cl_store(uint32_t a, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

// one cluster of cs CTAs; attr: room for two attributes
inline cudaLaunchConfig_t cluster_config(int cs, int threads, size_t smem, cudaStream_t st, cudaLaunchAttribute* attr,
                                         bool pdl) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 2 : 1;
    return cfg;
}

// opt-ins of a cluster kernel on the current device; false if it cannot run there
template <typename K>
bool cluster_prepare(K k, const cudaLaunchConfig_t& cfg) {
    int num = 0;
    const bool ok =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes) == cudaSuccess &&
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&num, k, &cfg) == cudaSuccess && num > 0;
    if (!ok) cudaGetLastError();
    return ok;
}

// the grids of the resident kernels: 64 to 256 points per axis, up to 2^15 points (spectral stages: 2^14)
#define RS_CASE(L1, L2, ...) \
    case (L1)*16 + (L2): { constexpr int B1 = L1, B2 = L2; __VA_ARGS__; } break;
#define RS_SP_CASES(...)                                                                      \
    RS_CASE(6, 6, __VA_ARGS__) RS_CASE(6, 7, __VA_ARGS__) RS_CASE(6, 8, __VA_ARGS__)          \
    RS_CASE(7, 6, __VA_ARGS__) RS_CASE(7, 7, __VA_ARGS__) RS_CASE(8, 6, __VA_ARGS__)
#define RS_DISPATCH(L1, L2, ...)                                                              \
    switch ((L1)*16 + (L2)) {                                                                 \
        RS_SP_CASES(__VA_ARGS__) RS_CASE(7, 8, __VA_ARGS__) RS_CASE(8, 7, __VA_ARGS__)        \
        default: break;                                                                       \
    }
#define RS_SP_DISPATCH(L1, L2, ...)                                                           \
    switch ((L1)*16 + (L2)) {                                                                 \
        RS_SP_CASES(__VA_ARGS__)                                                              \
        default: break;                                                                       \
    }
