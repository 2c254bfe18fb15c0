// Launches of the kernels that follow one another on a register's state.
//
// A kernel launched with launch_chained may be brought onto the SMs while the
// one before it on the stream still runs (programmatic dependent launch, also
// inside captured graphs): its launch latency and its prologue overlap the
// other's tail.  Such a kernel calls chain_wait() before it touches the state
// (it returns once every earlier kernel of the stream has completed and its
// writes are visible), and chain_release() as early as the next kernel may
// come onto the SMs: at its start, or, if it allocates TMEM, after that (the
// next kernel's blocks must not take TMEM that this kernel's still need).
// Kernels and copies launched without the attribute wait for completion as
// usual.  Only states that fit the L2 cache are chained: on large
// ones the latency is nothing against the pass (direct gate calls on 4.3e8
// amplitudes 10.80 ms chained, 10.62 not).  Measured: 500 gates on 4.8e6 complex64 amplitudes in L2 3747 -> 3567
// us; 40 gates on 324 complex128 amplitudes, planned, run and read, 497 -> 398 us.
#pragma once
#include <cstdint>
#include <utility>

#include <cuda_runtime.h>

namespace qd {

__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

constexpr uint64_t kChainBytes = uint64_t(128) << 20;

// state_bytes: the size of the state the kernel works on.
template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*fn)(P...), int grid, int block, size_t smem, cudaStream_t s, uint64_t state_bytes,
                                  A &&...args) {
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = s && state_bytes <= kChainBytes ? 1 : 0;  // (the legacy default stream orders whole kernels)
    return cudaLaunchKernelEx(&c, fn, std::forward<A>(args)...);
}

}  // namespace qd
