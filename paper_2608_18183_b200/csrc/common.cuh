// Device helpers shared by the kernels of the rollout library.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdlib>
#include <utility>

namespace hbsjd {

typedef __nv_bfloat16 bf16;

// Programmatic dependent launch: every kernel of the library has a pdl_wait() (blocks until the preceding
// grid in the stream has completed and its writes are visible) and a pdl_trigger() (lets the next grid's
// CTAs be scheduled as SMs free up), so launch latency and kernel prologues overlap the previous kernel's
// tail.  Most trigger after their own wait ("late"): triggered before it, a third kernel's CTAs take the shared memory
// that the second's would have had (one L image 0.94 times the time with the gate/up projection late, 24 L images token
// by token 0.99, four tiny images 0.99 with the small kernels late).
// All that precedes a late kernel is complete when the next one starts.  Four kernels use that: the QKV projection (rows,
// pages and rotations), attention (work list, pages, old keys), the accept kernel behind an LM head and k_commit read what
// kernels before their predecessor have written before their own wait, through L2.  Else nothing before pdl_wait() touches
// global memory that any kernel writes.  Stream carries which kind the last kernel was: the launchers of these four hand it
// to the kernel, which waits first behind a kernel that triggers early.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A stream and how the kernel launched there last triggers its successor.
struct Stream {
    cudaStream_t s;
    bool late;  // after its own wait; false too where it is not known (the first launch of a call)
    Stream(cudaStream_t stream) : s(stream), late(false) {}
    operator cudaStream_t() const { return s; }
};

// cluster_x > 1 launches thread-block clusters of that many CTAs along x.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kc(bool late, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, Stream& s,
                             int cluster_x, Args&&... args) {
    s.late = late;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    int n = 0;
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
    if (cluster_x > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster_x;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// For kernels that trigger after their own wait; launch_early for the others.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, Stream& s, Args&&... args) {
    return launch_kc(true, kernel, grid, block, smem, s, 1, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_early(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, Stream& s, Args&&... args) {
    return launch_kc(false, kernel, grid, block, smem, s, 1, std::forward<Args>(args)...);
}

// Raises a kernel's dynamic shared-memory limit once per device (function attributes are per device).
template <typename K>
inline cudaError_t ensure_dynamic_smem(K kernel, int bytes, int (&configured)[64]) {
    int dev = 0;
    cudaGetDevice(&dev);
    dev &= 63;
    if (bytes > configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
        configured[dev] = bytes;
    }
    return cudaSuccess;
}

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<bf16>(bf16 v) { return __bfloat162float(v); }

template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f<bf16>(float v) { return __float2bfloat16_rn(v); }

// Philox4x32-10 keyed by the rollout seed; counter = (image, position, round, 0).
// word 0: accept uniform, 1: replacement / bonus sample, 2: draft refresh sample, 3: fallback draft token.
__host__ __device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                       uint32_t k0, uint32_t k1, uint32_t out[4]) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
        const uint32_t n1 = (uint32_t)p1;
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
        const uint32_t n3 = (uint32_t)p0;
        c0 = n0; c1 = n1; c2 = n2; c3 = n3;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Physical KV location of (cache row, sequence index) through the page table.
struct KvView {
    void* k;               // [L][n_pages][page][D]
    void* v;
    const int32_t* table;  // [rows][pages_per_row]
    int pages_per_row, page, n_pages, D;
    __device__ __forceinline__ size_t offset(int layer, int row, int s) const {
        const int pg = table[row * pages_per_row + s / page];
        return (((size_t)layer * n_pages + pg) * page + (s % page)) * (size_t)D;
    }
};

}  // namespace hbsjd
