// Launches of a time step's kernels as a chain (programmatic dependent launch):
// a kernel's CTAs are set up while the last CTAs of the one before still run,
// and wait there.  Every kernel launched so calls chain_wait() in every thread
// before it reads or writes what another kernel of the chain writes or reads
// (so that its own end implies the end of all before it), and chain_go() after
// that.  Data that earlier kernels of the chain write are not read by __ldg, which
// may be moved above the wait.
#pragma once

#include <utility>

#include <cuda_runtime.h>

namespace poro {

// the kernels before this one have finished, and their writes are visible
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// the next kernel may be set up once every CTA of this one has come here
__device__ __forceinline__ void chain_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// The predictor and the faces let the next kernel in early up to degree 3, where
// elements are short: a cycle of 384 elements at N = 2 takes 41.3 instead of 43.4
// microseconds, 12,288 elements in three clusters at N = 3 14.02 instead of 14.10 ms
// a pass.  Above, the early CTAs crowd the SMs that run out first.  Microseconds a step
// of 384 and 6,000 elements, early and late: N = 4 binary64 95.1, 912 and 95.5, 911,
// double-binary32 72.0, 508 and 69.0, 504; N = 5 158.2, 1,615 and 140.2, 1,613, 94.6,
// 905 and 88.3, 899; N = 6, 5,184 elements, four steps in double-binary32, 6.02 and 5.97 ms.
constexpr bool chain_early(int N) { return N <= 3; }

template <class... Params, class... Args>
cudaError_t launch_chained(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, void* stream,
                           Args&&... args) {
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
    if (err != cudaSuccess) cudaGetLastError();  // reported here, not by a later call
    return err;
}

}  // namespace poro
