// Shared device/host helpers of the SAGE hot-path kernels (sm_100a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sage.h"

namespace sage {

constexpr int kHeadDim = 128;
constexpr int kPageSize = 64;

// First data-dependent error wins; kernels keep going on safe values or return early.
__device__ __forceinline__ void report_status(int32_t* status, int code) {
    if (status != nullptr) atomicCAS(status, 0, code);
}

// Ancestor-or-self bitset of node i of a tree with n nodes (local parent indices).
// Returns 0 and sets *bad when the parent chain breaks the tree rules
// (root = node 0 with parent -1; every other node has 0 <= parent < index).
__device__ __forceinline__ uint64_t ancestor_bits(const int32_t* __restrict__ parent, int n, int i, bool* bad) {
    uint64_t a = 0;
    int cur = i;
    for (int it = 0; it < SAGE_MAX_NODES && cur >= 0; ++it) {
        a |= 1ull << cur;
        int par = parent[cur];
        if (cur == 0) {
            if (par != -1) *bad = true;
            break;
        }
        if (par < 0 || par >= cur) {
            *bad = true;
            break;
        }
        cur = par;
    }
    return a;
}

// Every kernel (but for merges that launch_in_order is for) is launched to overlap its launch with the end of the kernel before it
// (programmatic stream serialization), and all start with after_previous_kernel(): it waits there until that kernel has completed and its
// writes are visible, before it touches global memory, and then lets the next kernel of the stream be brought up.
// No block leaves without passing it: a kernel waits for its direct predecessor only, and that one's end has to mean that
// its own predecessor has ended.
// The split schedule's merge pays for it (0.4 us of a layer's 9 at 2k keys: the loads that find its work used to run before the
// wait), but what a kernel reads ahead of it need not be visible yet.
// Between dependent kernels of a few microseconds this hides most of the gap: eight levels of tree growth
// (sixteen sequences) and the history update 45 -> 33 us.
__device__ __forceinline__ void after_previous_kernel() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... Params, typename... Args>
inline cudaError_t launch(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, int cluster,
                          const Args&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 0 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// The same without the overlap: the kernel is brought up once the one before it has ended, with the whole chip to spread over.
template <typename... Params, typename... Args>
inline cudaError_t launch_in_order(void (*kernel)(Params...), dim3 grid, int threads, cudaStream_t stream, const Args&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = stream;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

// A call's result as the entry points return it.  The runtime also keeps a failure as the thread's last error: it is taken
// away here, so that no later call can mistake it for its own.
inline bool succeeded(cudaError_t e) {
    if (e == cudaSuccess) return true;
    (void)cudaGetLastError();
    return false;
}
inline int launch_status(cudaError_t e) { return succeeded(e) ? SAGE_OK : SAGE_ERR_CUDA; }

}  // namespace sage
