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
// usual.
//
// Chaining pays where a launch is mostly latency, and costs where the early
// blocks take issue slots from the pass still running.  Per gate, 40 gates of
// one kind on complex64 states, unchained -> chained, us:
//   amplitudes      1 Ki          16 Ki         128 Ki        1 Mi        4 Mi
//   X,  D = 2   1.56 -> 1.35  1.58 -> 1.50  1.76 -> 1.90  3.05 -> 2.94  7.14 -> 7.41
//   X,  D = 3   1.69 -> 1.45  1.75 -> 1.61  2.13 -> 2.14  4.54 -> 4.30 10.12 -> 10.17 (177 Ki, 1.6, 4.8 Mi)
//   Z,  D = 3   1.92 -> 1.48  1.96 -> 1.62  2.10 -> 2.08  4.15 -> 3.79  8.62 -> 8.36 (the same)
//   dense D = 3 1.71 -> 1.35  1.71 -> 1.47  1.76 -> 1.60  2.85 -> 2.63  6.61 -> 6.38
//   dense D = 4 1.86 -> 1.51  1.91 -> 1.61  1.96 -> 1.99  3.92 -> 3.87 10.23 -> 9.98 (256 Ki: 2.12 -> 2.82)
//   dense D = 8 2.17 -> 1.71  2.64 -> 2.18  2.68 -> 2.67  5.09 -> 4.42
//   D = 10, tensor cores      3.92 -> 3.65  3.96 -> 3.66  6.73 -> 6.49 13.26 -> 12.92
// So every kernel chains on states of kChainBytes; complex64 gates of three
// states, dense or not, which gain or tie at every size (those of two and four
// lose at 64 to 256 Ki, and complex128 ones at 128 Ki: 2.6 -> 3.7), and the
// tensor-core kernels (qd_tc64.cu has an exception) on all states that fit L2
// (kChainL2Bytes; on larger ones it is a loss: direct gate calls on 4.3e8
// amplitudes 10.80 ms chained, 10.62 not); and the CUDA-core dense kernels above 8 states never (D = 9:
// 3.65 -> 3.73 at 16 Ki, 3.61 -> 4.43 at 256 Ki, 4.64 -> 7.01 at 1 Mi).
// 40 gates on 324 complex128 amplitudes, planned, run and read: 497 -> 398 us.
#pragma once
#include <cstdint>
#include <utility>

#include <cuda_runtime.h>

namespace qd {

__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

constexpr uint64_t kChainBytes = uint64_t(256) << 10;
constexpr uint64_t kChainL2Bytes = uint64_t(128) << 20;

// state_bytes: the size of the state the kernel works on; limit: up to which
// it is chained (0: never).
template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*fn)(P...), int grid, int block, size_t smem, cudaStream_t s, uint64_t state_bytes, uint64_t limit,
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
    c.numAttrs = s && state_bytes <= limit ? 1 : 0;  // (the legacy default stream orders whole kernels)
    return cudaLaunchKernelEx(&c, fn, std::forward<A>(args)...);
}

}  // namespace qd
