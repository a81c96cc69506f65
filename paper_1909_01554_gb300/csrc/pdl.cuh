// Programmatic dependent launch. A kernel that launch_pdl launches may start
// before its predecessor in the stream has ended, so each of its threads calls
// wait_for_operands first, which returns when the whole predecessor, and so everything
// older, has ended and its writes are visible. dependents_may_launch then lets
// the next kernel's blocks take their places as this one's blocks leave. No
// parameter that points to a matrix may be __restrict__, read or written: the
// qualifier lets the compiler move its loads and stores across the wait.
//
// Launched in plain stream order, kernels of one stream followed each other on a
// tick of 2.05 us on this device (calls took 6.1, 8.2, 10.2, 12.3 us), and the
// tensor kernel's setup (barriers, TMEM, cluster: 1920 cycles) came after the
// pass that writes its operands. Measured, us a call back to back, plain order ->
// so: Boolean 2112 x 1984 x 2240 17.9 -> 10.9; one launch each, 256 x 512 x 384
// 6.1 -> 4.4, transpose 16448 x 12224 16.2 -> 13.3. The tensor kernel itself does
// not let the next one in early: blocks that wait beside it cost it more than
// they gain (4096^3 21.4 -> 26.7).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace bmm {

__device__ __forceinline__ void dependents_may_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_operands() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launches `kernel`, which calls wait_for_operands, behind the stream's last one.
template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem,
                       cudaStream_t s, A&&... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
    return e == cudaSuccess ? e : cudaGetLastError();  // (which clears it)
}

}  // namespace bmm
