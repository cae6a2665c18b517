// Kernel launches of the product path.
//
// Every product kernel is launched with programmatic stream serialisation:
// the kernel lets the next kernel of its stream be scheduled as soon as all
// of its own CTAs are running (griddepcontrol.launch_dependents at entry, or
// right after the allocation of tensor memory),
// and the next kernel runs its prologue -- barrier set-up, fetching the
// handle's own schedule and block values -- on the SMs that free up, then
// waits (griddepcontrol.wait) before it touches anything an earlier kernel
// may write: X, the bias, Y and the split-row workspace. A chain of products
// on one stream (layers, or the block-shape sweep) thus overlaps each
// kernel's start with the previous one's tail, with the stream's ordering
// intact. BSR_PDL=0 in the environment turns it off (plain stream order).
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <cstdlib>
#include <mutex>
#include <utility>

namespace bsr {

inline bool pdl_enabled() {
    static const bool on = [] {
        const char *v = std::getenv("BSR_PDL");
        return !(v && v[0] == '0');
    }();
    return on;
}

// cuTensorMapEncodeTiled (nullptr where the driver has none).
inline PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

// Lets `kernel` take `bytes` of dynamic shared memory on the current device;
// `done` keeps a bit per device that has it.
template <typename K>
cudaError_t allow_smem(K kernel, int bytes, std::atomic<uint64_t> &done) {
    int dev = 0;
    cudaGetDevice(&dev);
    const uint64_t bit = 1ull << (dev & 63);
    if (done.load() & bit) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit);
    return e;
}

// Launch `kernel` on `s` in clusters of `cluster` CTAs (1: no clusters).
template <typename... KArgs, typename... Args>
cudaError_t launch_clusters(void (*kernel)(KArgs...), unsigned cluster, dim3 grid, dim3 block, size_t smem,
                            cudaStream_t s, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (pdl_enabled()) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        n++;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster;
        attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
        n++;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Launch `kernel` on `s`.
template <typename... KArgs, typename... Args>
cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                          Args &&...args) {
    return launch_clusters(kernel, 1, grid, block, smem, s, std::forward<Args>(args)...);
}

}  // namespace bsr
