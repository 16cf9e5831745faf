// Plain arithmetic that kernels and launchers share and that a test can compile and check on its own: no CUDA in here.
#pragma once

#ifdef __CUDACC__
#define FC_RULE __host__ __device__ constexpr
#else
#define FC_RULE constexpr
#endif

namespace fc {

// How often slot `slot` of a ring of `slots` buffers has been asked for when `requested` boxes were requested in order.
// The barrier of a slot completes one phase per request, so the last one is phase ring_uses - 1.
FC_RULE int ring_uses(long long requested, int slot, int slots) {
    return requested > slot ? (int)((requested - slot + slots - 1) / slots) : 0;
}

}  // namespace fc
