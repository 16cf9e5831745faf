// Programmatic dependent launch for the kernels of a pass.
//
// A pass is three kernels in one stream (forward transforms, contraction, inverse
// transform) and a training step is nine.  Launched the plain way, each kernel starts
// only after its predecessor has drained completely, so every boundary costs a launch
// latency plus the kernel's own prologue (barrier setup, tensor-memory allocation).
// With the stream-serialization attribute the next grid may be scheduled while the
// previous one drains: its CTAs run their prologue and then block in dep_wait() until
// the previous grid has completed and its writes are visible.  Every kernel calls
// dep_wait() before its first global-memory access (reads AND writes: a kernel may
// overwrite workspace that its predecessor still reads), so results are those of the
// serial order.  Without the attribute both device calls are no-ops.
#pragma once

#include <cuda_runtime.h>
#include <utility>

namespace fc {

// Allow the next kernel in the stream to be scheduled as soon as resources free up.
__device__ __forceinline__ void dep_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Block until every kernel this launch depends on has completed and flushed its writes.
__device__ __forceinline__ void dep_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// `overlap` = false launches the plain way.  Where overlapping pays was measured on B200
// (three layer configurations and a 1,000-point sweep of the parameter grid):
//  * contraction after one-pass forward transforms, inverse transform after the contraction:
//    1-7 % shorter passes at n <= 64 with the tensor-core contraction (the two-team inverse of n = 64 excepted, see
//    fft_inv64.cuh: a dependent's CTAs lose the placement that lets neighbours share sectors);
//  * the forward transforms as dependents of the previous pass's inverse transform gain
//    nothing at n <= 32, and at n = 64 a training step took 1.14 ms instead of 0.74;
//  * at n = 128 a pass is 0.5 % longer with the contraction as a
//    dependent and 2.5 % longer with the inverse transform as one (2-6 % over the sweep);
//  * the FP32 contractions only where the sum is one k-block of 16 (2 us shorter passes, 24 -> 21 us on
//    an S8 f4 f'8 16 x 16 layer).  While the transforms drain, the CTAs of a dependent (128 threads) pile up four to
//    an SM on the few SMs that are free, and a longer chain of k-blocks then runs at a fourth of its pace:
//    FP32 passes at n = 8, S16 f64 f'64 fprop 15.6 -> 29.6 us against 16.5 on its own, at n = 32 S4 f256 f'64
//    fprop 151 against 79.  Of 309 FP32 passes (n = 8 .. 64) 15 are up to 14 % (2 us) shorter as dependents all the
//    same, most of them with sums of 32 to 64;
//  * the inverse transform after an FP32 contraction, whatever its sum: 1-3 us shorter passes.
// The callers set the flag accordingly; everything else is launched the plain way.
struct DepConfig {
    bool overlap;
    int cluster;                // CTAs per cluster
    // Percentage of an SM's L1 asked for as shared memory, -1: as the kernel's footprint has it.  An SM changes that division
    // only when it is idle, so a kernel with a small footprint between kernels with a large one starts late and ends
    // the overlap with its neighbours: 1 - 4 us per pass of 12 - 25 us.  (Not for every kernel: the forward transforms
    // read their samples through the L1, wide planes 1713 -> 1923 us with all of it shared memory.)
    int carveout;
    DepConfig(bool overlap_, int cluster_ = 1, int carveout_ = -1) : overlap(overlap_), cluster(cluster_), carveout(carveout_) {}
};
template <typename... KArgs, typename... Args>
static cudaError_t dep_launch(DepConfig c, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[3];
    int n = 0;
    if (c.overlap) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (c.cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)c.cluster;
        attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (c.carveout >= 0) {
        attr[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        attr[n++].val.sharedMemCarveout = (unsigned)c.carveout;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

}  // namespace fc
