// Programmatic dependent launch: the pass that writes a tensor kernel's
// operands lets that kernel's blocks start while it still runs
// (dependents_may_launch, once all its own blocks run), and the tensor kernel
// waits for the whole pass before it reads them (wait_for_operands). Launch and
// setup of the tensor kernel (barriers, TMEM, cluster: 1920 cycles) then overlap
// the pass. A pass itself is launched in stream order, so nothing older than the
// pass can still run. Measured (us a product, before -> now): GF(2) 256 x 512 x
// 384 8.9 -> 6.9 and 4096^3 24.2 -> 22.9 inside a graph; Boolean 2112 x 1984 x
// 2240 17.9 -> 14.3 and a batch of 512 small products 43.1 -> 39.3 as calls.
#pragma once

namespace bmm {

__device__ __forceinline__ void dependents_may_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_operands() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace bmm
