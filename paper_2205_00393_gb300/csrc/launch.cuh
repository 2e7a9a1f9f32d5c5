// Programmatic dependent launches. A kernel launched with launch_dependent may
// start while its predecessor in the stream still runs, once every CTA of that one
// has called dep_trigger() or ended; dep_wait() then waits until the predecessor
// has completed and its writes are visible. Before it, a kernel only reads its
// parameters and the tables that the host uploaded (a copy in the stream is a full
// dependency): decoding them hides behind the predecessor's last CTAs, together
// with the launch itself. Every CTA of a kernel that is launched this way calls
// dep_wait() before it ends, so that its completion implies its predecessor's.
// Data that a predecessor writes is read through plain pointers: a load through
// the read-only path (__ldg) or a __restrict__ pointer, of which nothing else is
// supposed to write the target, may be moved above the wait. __restrict__ is for the
// uploaded tables.
//
// dep_trigger() in a kernel lets its successor start early. That pays for short
// kernels and costs in long ones, whose successor's waiting CTAs take places and
// issue slots from them: kernels of up to two or three waves call it, the others (and the
// stem and CTA-pair kernels) leave it to their CTAs' ends, which still hides the
// launch. The 27 launches of a 20-qubit split BF16 call take 237 us one after
// another, 180 without and 161 with early triggers; a 25-qubit split TF32 call
// 5.92 ms, 5.55 without, 5.80 with them everywhere, and a 28-qubit stem 75.2 ms,
// 75.2 and 78.9.
#pragma once

#include <cuda_runtime.h>

namespace tnc {

constexpr unsigned kTriggerCtas = 1216;  // 152 SMs x 8: two waves at four CTAs per SM, 2.7 at the grouped FP32 kernels' three
__device__ __forceinline__ void dep_trigger() {
    if (gridDim.x * gridDim.y * gridDim.z <= kTriggerCtas) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// cluster > 1: CTAs per cluster (x), for kernels without a cluster shape of their own
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2]{};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace tnc
