// Register initialisation and FP64 readout kernels (QuDiet Sec. 3.2
// init_states; Sec. 3.8 output as amplitudes or probabilities), plus the
// measurement-sampling extension (prefix sums of probabilities and inverse-CDF
// draws from a counter-based generator).
//
// Every reduction accumulates in FP64 in a fixed order (per-thread strided
// sums, then a fixed tree), so results are run-to-run deterministic.
#include <cstdint>
#include <cuda_runtime.h>

#include "qd_common.cuh"
#include "qd_fixed.cuh"
#include "qd_launch.cuh"
#include "qd_reduce.h"

namespace qd {

namespace {

constexpr int kRedBlock = 256;

__device__ __forceinline__ double block_sum(double v, double *sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    v = 0.0;
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        v = lane < nw ? sh[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    return v;  // valid in thread 0
}

// psi = 0 except psi[idx] = 1.
template <typename T>
__global__ void k_init(v2<T> *psi, uint64_t N, uint64_t idx) {
    chain_release();
    chain_wait();
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += step)
        psi[i] = mk<T>(i == idx ? T(1) : T(0), T(0));
}

// Two consecutive amplitudes at an even index i (16-byte aligned complex64
// pairs), zeros beyond N.
template <typename T, bool ALIGNED = true>
__device__ __forceinline__ void load_pair(const v2<T> *__restrict__ psi, v2<T> *v) {
    if constexpr (sizeof(T) == 4 && ALIGNED) {
        const float4 q = *reinterpret_cast<const float4 *>(psi);
        v[0] = make_float2(q.x, q.y);
        v[1] = make_float2(q.z, q.w);
    } else {
        v[0] = psi[0];
        v[1] = psi[1];
    }
}
template <typename T, bool ALIGNED = true>
__device__ __forceinline__ void load_pair(const v2<T> *__restrict__ psi, uint64_t i, uint64_t N, v2<T> *v) {
    if (i + 1 < N) {
        load_pair<T, ALIGNED>(psi + i, v);
    } else {
        v[0] = i < N ? psi[i] : mk<T>(T(0), T(0));
        v[1] = mk<T>(T(0), T(0));
    }
}

// Amplitudes per thread and iteration of the sums below: the loads in flight
// (64 bytes a thread) and the group whose squares are added on the integer
// units (qd_fixed.cuh).  (Two of ten complex64 amplitudes on the FP64 pipe
// beside them made it the limit: the norm of 3.4e8 took 644 us, not 508.)
template <typename T> constexpr int kSumGroup = sizeof(T) == 4 ? 8 : 4;

// Per-block partial sums of |psi_i|^2 over the whole state.  Bound by the
// read of the state: 16-byte loads, one FP64 addition per group of 8 (4)
// amplitudes.  With both squares of every amplitude in FP64 (conversions
// included, five operations of the FP64 pipe each) the pipe's two lanes per
// SM took 6x the time of the read on complex64 states.  3.4e8 amplitudes:
// complex64 3154 -> 494 us (5.5 TB/s), complex128 1923 -> 868 us (6.26).
template <typename T>
__global__ void __launch_bounds__(kRedBlock, 5) k_norm_partial(const v2<T> *__restrict__ psi, uint64_t N,
                                                            double *__restrict__ part) {
    __shared__ double sh[32];
    constexpr int G = kSumGroup<T>;
    const uint64_t tile = (uint64_t)G * kRedBlock;
    double acc = 0.0;
    for (uint64_t t = (uint64_t)blockIdx.x * tile; t < N; t += (uint64_t)gridDim.x * tile) {
        v2<T> v[G];
        if (t + tile <= N) {
            const v2<T> *p = psi + t + 2 * threadIdx.x;
#pragma unroll
            for (int k = 0; k < G / 2; ++k) load_pair<T>(p + 2 * k * kRedBlock, v + 2 * k);
        } else {
#pragma unroll
            for (int k = 0; k < G / 2; ++k) load_pair<T>(psi, t + 2 * (k * kRedBlock + threadIdx.x), N, v + 2 * k);
        }
        acc += group_norm<T, G>(v);
    }
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// Partial sums per digit of a low qudit (stride s, dimension d, period P = s d
// of at most kPeriodMax): the first A threads of the grid (a multiple of P)
// walk the state with step A, so that a thread meets one digit only and a
// warp's loads are consecutive; every amplitude is read once.  One block sum
// per digit at the end, hence only up to kPeriodDim levels.  3.4e8 complex64
// amplitudes: 3248 -> 524 us (5.2 TB/s; 584 with bounds checks in full tiles).
constexpr uint32_t kPeriodMax = 16384;
constexpr int kPeriodDim = 8;

template <typename T>
__global__ void __launch_bounds__(kRedBlock, 5) k_digit_partial(const v2<T> *__restrict__ psi, uint64_t N, uint32_t s,
                                                             uint32_t d, uint32_t A, double *__restrict__ part) {
    __shared__ double sh[32];
    constexpr int G = kSumGroup<T>;
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
    double acc = 0.0;
    if (tid < A) {
        for (uint64_t i = tid; i < N; i += (uint64_t)G * A) {
            v2<T> v[G];
            if (i + (uint64_t)(G - 1) * A < N) {
                const v2<T> *p = psi + i;
#pragma unroll
                for (int k = 0; k < G; ++k, p += A) v[k] = *p;
            } else {
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    const uint64_t j = i + (uint64_t)k * A;
                    v[k] = j < N ? psi[j] : mk<T>(T(0), T(0));
                }
            }
            acc += group_norm<T, G>(v);
        }
    }
    const uint32_t digit = (tid / s) % d;
    for (uint32_t x = 0; x < d; ++x) {
        const double b = block_sum(digit == x && tid < A ? acc : 0.0, sh);
        if (threadIdx.x == 0) part[(size_t)x * gridDim.x + blockIdx.x] = b;
    }
}

// Partial sums of the digit slices of a qudit with runs of s amplitudes: the
// blocks of slice y walk its M = N / d amplitudes in order, r = q s + l at
// index q P + y s + l.  LONG (s at least a block's tile, which then meets at
// most two runs): one division per tile instead of one per amplitude, whose
// operations share the ALU pipe with the squares'.  3.4e8 complex64
// amplitudes: 3245 us with FP64 squares, 784 with a division per amplitude,
// 672 with LONG and 473 to 494 (5.6 TB/s) without bounds checks in full tiles.
template <typename T, bool LONG>
__global__ void __launch_bounds__(kRedBlock, 5) k_slice_partial(const v2<T> *__restrict__ psi, uint64_t M,
                                                                FastDiv64 divs, uint64_t P,
                                                                double *__restrict__ part) {
    __shared__ double sh[32];
    constexpr int G = kSumGroup<T>;
    const uint64_t s = divs.d, off = (uint64_t)blockIdx.y * s, skip = P - s;
    const uint64_t tile = (uint64_t)G * kRedBlock;
    double acc = 0.0;
    for (uint64_t t = (uint64_t)blockIdx.x * tile; t < M; t += (uint64_t)gridDim.x * tile) {
        v2<T> v[G];
        const uint64_t q = LONG ? fdiv(t, divs) : 0;
        const uint64_t left = LONG ? s - (t - q * s) : 0;  // of the tile's first run
        const v2<T> *first = psi + t + q * skip + off;
        if (LONG && left >= tile && t + tile <= M) {  // one run
#pragma unroll
            for (int k = 0; k < G; ++k) v[k] = first[k * kRedBlock + threadIdx.x];
        } else
#pragma unroll
        for (int k = 0; k < G; ++k) {
            const uint32_t e = k * kRedBlock + threadIdx.x;
            const uint64_t r = t + e;
            if constexpr (LONG) v[k] = r < M ? first[e + (e >= left ? skip : 0)] : mk<T>(T(0), T(0));
            else v[k] = r < M ? psi[r + fdiv(r, divs) * skip + off] : mk<T>(T(0), T(0));
        }
        acc += group_norm<T, G>(v);
    }
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) part[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = acc;
}

// out[y] = sum over the nb partials of slice y, in index order per thread.
__global__ void k_sum_partials(const double *__restrict__ part, int nb, double *__restrict__ out) {
    __shared__ double sh[32];
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) acc += part[(size_t)blockIdx.x * nb + i];
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) out[blockIdx.x] = acc;
}

// Per-block partial sums of conj(a_i) * b_i, fixed order.  Bound by the two
// reads: groups of four products are added on the integer units
// (qd_fixed.cuh), two FP64 additions per group.  In FP64 the conversions and
// products are eight operations of its pipe per complex64 pair.  3.4e8
// amplitudes: complex64 pairs 5098 -> 1850 us, complex64 with complex128
// 3882 -> 1806 us (4.5 TB/s; 2014 without the FP64 pipe's share), complex128
// pairs 2416 -> 2056 us (5.3 TB/s; 2390); the ALU pipe is the limit now (139
// instructions per mixed pair).
template <typename TA, typename TB>
__global__ void __launch_bounds__(kRedBlock) k_overlap_partial(const v2<TA> *__restrict__ a, const v2<TB> *__restrict__ b,
                                                               uint64_t N, double *__restrict__ part) {
    __shared__ double sh[32];
    // a group on the integer units and, with a complex128 state (no or half the
    // conversions), two pairs on the FP64 pipe beside it
    constexpr int G = 4, F = sizeof(TA) + sizeof(TB) > 8 ? 2 : 0;
    const uint64_t tile = (uint64_t)(G + F) * kRedBlock;
    double re = 0.0, im = 0.0;
    for (uint64_t t = (uint64_t)blockIdx.x * tile; t < N; t += (uint64_t)gridDim.x * tile) {
        v2<TA> x[G + F];
        v2<TB> y[G + F];
        if (t + tile <= N) {
            const v2<TA> *pa = a + t + 2 * threadIdx.x;
            const v2<TB> *pb = b + t + 2 * threadIdx.x;
#pragma unroll
            for (int k = 0; k < (G + F) / 2; ++k) {
                load_pair<TA>(pa + 2 * k * kRedBlock, x + 2 * k);
                load_pair<TB>(pb + 2 * k * kRedBlock, y + 2 * k);
            }
        } else {
#pragma unroll
            for (int k = 0; k < (G + F) / 2; ++k) {
                const uint64_t i = t + 2 * (k * kRedBlock + threadIdx.x);
                load_pair<TA>(a, i, N, x + 2 * k);
                load_pair<TB>(b, i, N, y + 2 * k);
            }
        }
        double gr, gi;
        group_overlap<TA, TB, G>(x, y, gr, gi);
        re += gr;
        im += gi;
#pragma unroll
        for (int k = G; k < G + F; ++k) {
            const double xr = (double)x[k].x, xi = (double)x[k].y, yr = (double)y[k].x, yi = (double)y[k].y;
            re = fma(xr, yr, fma(xi, yi, re));
            im = fma(xr, yi, fma(-xi, yr, im));
        }
    }
    re = block_sum(re, sh);
    im = block_sum(im, sh);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = re;
        part[2 * blockIdx.x + 1] = im;
    }
}

__global__ void k_sum_pairs(const double *__restrict__ part, int nb, double *__restrict__ out) {
    __shared__ double sh[32];
    double re = 0.0, im = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        re += part[2 * i];
        im += part[2 * i + 1];
    }
    re = block_sum(re, sh);
    im = block_sum(im, sh);
    if (threadIdx.x == 0) {
        out[0] = re;
        out[1] = im;
    }
}

// p[i] = |psi_i|^2.  Bound by the read and the FP64 write: two amplitudes per
// thread and step (16-byte loads and stores), one FP64 addition per complex64
// amplitude (qd_fixed.cuh) instead of four operations of that pipe.  3.4e8
// complex64 amplitudes: 2531 -> 911 us (5.97 TB/s).
template <typename T, bool PAIRS>
__global__ void __launch_bounds__(kRedBlock) k_probs(const v2<T> *__restrict__ psi, uint64_t N, double *__restrict__ p) {
    if constexpr (PAIRS) {
        constexpr int U = 2;
        const uint64_t tile = 2 * U * kRedBlock;
        for (uint64_t t = (uint64_t)blockIdx.x * tile; t < N; t += (uint64_t)gridDim.x * tile) {
            v2<T> v[2 * U];
#pragma unroll
            for (int k = 0; k < U; ++k) load_pair<T>(psi, t + 2 * (k * kRedBlock + threadIdx.x), N, v + 2 * k);
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint64_t i = t + 2 * (k * kRedBlock + threadIdx.x);
                if (i + 1 < N) *reinterpret_cast<double2 *>(p + i) = make_double2(prob_of(v[2 * k]), prob_of(v[2 * k + 1]));
                else if (i < N) p[i] = prob_of(v[2 * k]);
            }
        }
    } else {  // an output that is not 16-byte aligned
        const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
        for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += step) p[i] = prob_of(psi[i]);
    }
}

// ---- prefix sums: chunk sums, scan of chunk sums, scan inside chunks -------
constexpr int kScanBlock = 256;
constexpr int kScanPer = 16;
constexpr int kChunk = kScanBlock * kScanPer;  // 4096 amplitudes per chunk

template <typename T, bool ALIGNED>
__global__ void __launch_bounds__(kScanBlock) k_chunk_sums(const v2<T> *__restrict__ psi, uint64_t N,
                                                           double *__restrict__ sums) {
    __shared__ double sh[32];
    const uint64_t c0 = (uint64_t)blockIdx.x * kChunk;
    constexpr int G = kSumGroup<T>;
    double acc = 0.0;
#pragma unroll
    for (int k0 = 0; k0 < kScanPer; k0 += G) {
        v2<T> v[G];
#pragma unroll
        for (int k = 0; k < G / 2; ++k)
            load_pair<T, ALIGNED>(psi, c0 + 2 * ((uint64_t)(k0 / 2 + k) * kScanBlock + threadIdx.x), N, v + 2 * k);
        acc += group_norm<T, G>(v);
    }
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0) sums[blockIdx.x] = acc;
}

// Exclusive scan of nb chunk sums in one block of 1024 threads; thread t owns
// a contiguous run.  Also writes the grand total to sums[nb].
__global__ void __launch_bounds__(1024) k_scan_sums(double *sums, uint64_t nb) {
    __shared__ double sh[1024];
    const uint64_t per = (nb + blockDim.x - 1) / blockDim.x;
    const uint64_t a = threadIdx.x * per, b = (a + per < nb) ? a + per : nb;
    double loc = 0.0;
    for (uint64_t i = a; i < b; ++i) loc += sums[i];
    sh[threadIdx.x] = loc;
    __syncthreads();
    // Hillis-Steele inclusive scan of the 1024 thread totals
    for (int o = 1; o < 1024; o <<= 1) {
        const double v = threadIdx.x >= (unsigned)o ? sh[threadIdx.x - o] : 0.0;
        __syncthreads();
        sh[threadIdx.x] += v;
        __syncthreads();
    }
    double run = threadIdx.x ? sh[threadIdx.x - 1] : 0.0;
    for (uint64_t i = a; i < b; ++i) {
        const double v = sums[i];
        sums[i] = run;
        run += v;
    }
    if (threadIdx.x == blockDim.x - 1) sums[nb] = sh[blockDim.x - 1];
}

// Shared-memory index with one pad entry per kScanPer, so the thread-serial
// pass (thread t owns entries t*kScanPer ...) does not hit one bank.
__device__ __forceinline__ int padx(int e) { return e + e / kScanPer; }

template <typename T>
__global__ void __launch_bounds__(kScanBlock) k_chunk_scan(const v2<T> *__restrict__ psi, uint64_t N,
                                                           const double *__restrict__ offs,
                                                           double *__restrict__ cdf) {
    __shared__ double buf[kChunk + kChunk / kScanPer];
    __shared__ double tot[kScanBlock];
    const uint64_t c0 = (uint64_t)blockIdx.x * kChunk;
    for (int k = 0; k < kScanPer; ++k) {
        const int e = k * kScanBlock + threadIdx.x;
        const uint64_t i = c0 + e;
        buf[padx(e)] = i < N ? prob_of(psi[i]) : 0.0;
    }
    __syncthreads();
    // each thread scans its kScanPer consecutive entries
    double run = 0.0;
    const int e0 = threadIdx.x * kScanPer;
    for (int k = 0; k < kScanPer; ++k) {
        run += buf[padx(e0 + k)];
        buf[padx(e0 + k)] = run;
    }
    tot[threadIdx.x] = run;
    __syncthreads();
    for (int o = 1; o < kScanBlock; o <<= 1) {
        const double v = threadIdx.x >= (unsigned)o ? tot[threadIdx.x - o] : 0.0;
        __syncthreads();
        tot[threadIdx.x] += v;
        __syncthreads();
    }
    const double add = offs[blockIdx.x] + (threadIdx.x ? tot[threadIdx.x - 1] : 0.0);
    for (int k = 0; k < kScanPer; ++k) buf[padx(e0 + k)] += add;
    __syncthreads();
    for (int k = 0; k < kScanPer; ++k) {
        const int e = k * kScanBlock + threadIdx.x;
        const uint64_t i = c0 + e;
        if (i < N) cdf[i] = buf[padx(e)];
    }
}

// ---- sampling ---------------------------------------------------------------
// Philox4x64-10 (Salmon et al., SC 2011): two 64x64->128 multiplies per round
// with the published multipliers and Weyl key increments.
__device__ __forceinline__ uint64_t philox_word0(uint64_t c0, uint64_t key0) {
    uint64_t c[4] = {c0, 0, 0, 0};
    uint64_t k0 = key0, k1 = 0;
    const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
    const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
        const uint64_t hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
        const uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
        k0 += W0;
        k1 += W1;
    }
    return c[0];
}

// Sampling draws shot s at the smallest i with CDF_i > u_s CDF_{N-1} without
// writing the CDF: the state is read once, and what is kept are prefix sums at
// three levels (16 amplitudes inside a chunk of 4096, chunks inside a super of
// 1024 chunks, supers), 1/2 byte per amplitude instead of a second read of the
// state and 8 bytes per amplitude written and read again.  A shot searches the
// levels from the top and walks its 16 amplitudes.  Every level's prefix is
// relative to its parent, and base + prefix > target decides at each.  One
// shot from 3.4e8 complex64 amplitudes: 7582 us with the whole CDF, 582 us
// (4.67 TB/s); a million shots: 8115 -> 850 us.
constexpr int kSampBlock = 256;
constexpr int kSampPer = 16;                       // amplitudes per prefix entry
constexpr int kSampChunk = kSampBlock * kSampPer;  // amplitudes per chunk
constexpr int kSampSuper = 1024;                   // chunks per super

// Inclusive scan of one value per thread over the block, thread order.
template <int THREADS>
__device__ __forceinline__ double block_incl_scan(double v, double *sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    __syncthreads();
    if (lane == 31) sh[w] = v;
    __syncthreads();
    double t = lane < THREADS / 32 ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 1; o < THREADS / 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += y;
    }
    const double before = __shfl_sync(0xffffffffu, t, w > 0 ? w - 1 : 0);
    return w > 0 ? v + before : v;
}

// One chunk: staged in shared memory by asynchronous 16-byte copies (rows of
// 16 amplitudes, one per thread, padded by 16 bytes: conflict-free 16-byte
// reads), so that the state's reads are coalesced although a thread sums
// consecutive amplitudes.
template <typename T> constexpr int kSampRow = kSampPer * (int)sizeof(v2<T>) + 16;

template <typename T>
__global__ void __launch_bounds__(kSampBlock) k_samp_prefix(const v2<T> *__restrict__ psi, uint64_t N,
                                                            double *__restrict__ pre, double *__restrict__ tot) {
    extern __shared__ __align__(16) unsigned char rows[];
    __shared__ double sh[32];
    constexpr int R16 = kSampPer * (int)sizeof(v2<T>) / 16;  // 16-byte pieces of a row
    constexpr int A16 = 16 / (int)sizeof(v2<T>);             // amplitudes of a piece
    const uint64_t c0 = (uint64_t)blockIdx.x * kSampChunk;
    if (c0 + kSampChunk <= N) {
#pragma unroll
        for (int k = 0; k < R16; ++k) {
            const int e = k * kSampBlock + threadIdx.x;
            const unsigned dst = (unsigned)__cvta_generic_to_shared(rows + (e / R16) * kSampRow<T> + (e % R16) * 16);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(psi + c0 + e * A16) : "memory");
        }
    } else {
#pragma unroll
        for (int k = 0; k < R16; ++k) {
            const int e = k * kSampBlock + threadIdx.x;
            const uint64_t i = c0 + (uint64_t)e * A16;
            // pieces beyond N (and the odd half of the last one) are filled with zeros
            const int bytes = i >= N ? 0 : (N - i >= A16 ? 16 : (int)sizeof(v2<T>));
            const unsigned dst = (unsigned)__cvta_generic_to_shared(rows + (e / R16) * kSampRow<T> + (e % R16) * 16);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(psi + (bytes ? i : 0)), "r"(bytes)
                         : "memory");
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    const float4 *row = reinterpret_cast<const float4 *>(rows + threadIdx.x * kSampRow<T>);
    constexpr int G = kSumGroup<T>;
    double s = 0.0;
#pragma unroll
    for (int g = 0; g < kSampPer / G; ++g) {
        v2<T> v[G];
#pragma unroll
        for (int q = 0; q < G / A16; ++q) {
            const float4 x = row[g * (G / A16) + q];
            if constexpr (sizeof(T) == 4) {
                v[2 * q] = make_float2(x.x, x.y);
                v[2 * q + 1] = make_float2(x.z, x.w);
            } else {
                v[q] = make_double2(__hiloint2double(__float_as_int(x.y), __float_as_int(x.x)),
                                    __hiloint2double(__float_as_int(x.w), __float_as_int(x.z)));
            }
        }
        s += group_norm<T, G>(v);
    }
    s = block_incl_scan<kSampBlock>(s, sh);
    pre[(uint64_t)blockIdx.x * kSampBlock + threadIdx.x] = s;
    if (threadIdx.x == kSampBlock - 1) tot[blockIdx.x] = s;
}

// Chunk totals -> inclusive prefix inside each super; super totals.
__global__ void __launch_bounds__(kSampSuper) k_samp_super(double *__restrict__ tot, uint64_t nchunks,
                                                           double *__restrict__ sup) {
    __shared__ double sh[32];
    const uint64_t c = (uint64_t)blockIdx.x * kSampSuper + threadIdx.x;
    const double v = block_incl_scan<kSampSuper>(c < nchunks ? tot[c] : 0.0, sh);
    if (c < nchunks) tot[c] = v;
    if (threadIdx.x == kSampSuper - 1) sup[blockIdx.x] = v;
}

// Super totals -> inclusive prefix (one block).
__global__ void __launch_bounds__(kSampSuper) k_samp_top(double *__restrict__ sup, uint64_t n) {
    __shared__ double sh[32];
    __shared__ double carry;
    if (threadIdx.x == 0) carry = 0.0;
    __syncthreads();
    for (uint64_t b = 0; b < n; b += kSampSuper) {
        const uint64_t i = b + threadIdx.x;
        const double v = block_incl_scan<kSampSuper>(i < n ? sup[i] : 0.0, sh) + carry;
        __syncthreads();
        if (i < n) sup[i] = v;
        if (threadIdx.x == kSampSuper - 1) carry = v;
        __syncthreads();
    }
}

// smallest k < n with base + a[k] > target, or n
__device__ __forceinline__ uint64_t first_above(const double *__restrict__ a, uint64_t n, double base, double target) {
    uint64_t lo = 0, hi = n;
    while (lo < hi) {
        const uint64_t mid = lo + ((hi - lo) >> 1);
        if (base + a[mid] > target) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}
// ... or, where the parent's prefix exceeds the target by less than the
// children's rounding, the first entry that reaches the children's total
__device__ __forceinline__ uint64_t descend(const double *__restrict__ a, uint64_t n, double &base, double target) {
    uint64_t k = first_above(a, n, base, target);
    if (k == n) {
        const double last = a[n - 1];
        uint64_t lo = 0, hi = n - 1;
        while (lo < hi) {
            const uint64_t mid = lo + ((hi - lo) >> 1);
            if (a[mid] >= last) hi = mid;
            else lo = mid + 1;
        }
        k = lo;
    }
    if (k > 0) base += a[k - 1];
    return k;
}

template <typename T>
__global__ void __launch_bounds__(256) k_samp_draw(const v2<T> *__restrict__ psi, uint64_t N,
                                                   const double *__restrict__ pre, const double *__restrict__ tot,
                                                   uint64_t nchunks, const double *__restrict__ sup, uint64_t nsup,
                                                   const double *__restrict__ u, uint64_t seed, int64_t shots,
                                                   int64_t *__restrict__ out) {
    const double total = sup[nsup - 1];
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < shots; s += (int64_t)gridDim.x * blockDim.x) {
        double us;
        if (u) {
            us = u[s];
        } else {
            us = (double)(philox_word0((uint64_t)s, seed) >> 11) * (1.0 / 9007199254740992.0);
        }
        const double target = us * total;
        uint64_t found = N - 1;  // u >= 1, or sums that are not numbers
        if (total > target) {
            double base = 0.0;
            const uint64_t p = descend(sup, nsup, base, target);
            const uint64_t cb = p * kSampSuper, cn = min((uint64_t)kSampSuper, nchunks - cb);
            const uint64_t c = cb + descend(tot + cb, cn, base, target);
            const uint64_t k = descend(pre + c * kSampBlock, kSampBlock, base, target);
            const uint64_t i0 = c * kSampChunk + k * kSampPer;
            found = i0 < N ? i0 : N - 1;
            double run = base;
            for (uint64_t i = i0; i < N && i < i0 + kSampPer; ++i) {
                const double q = prob_of(psi[i]);
                run += q;
                if (q > 0.0 || run > target) found = i;
                if (run > target) break;
            }
        }
        out[s] = (int64_t)found;
    }
}

int grid_for(uint64_t n, int block, int sm_count, int per_sm) {
    uint64_t g = (n + block - 1) / block;
    const uint64_t cap = (uint64_t)sm_count * per_sm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

}  // namespace

cudaError_t init_basis(void *psi, int prec, uint64_t N, uint64_t idx, int sm_count, cudaStream_t s) {
    const int g = grid_for(N, 256, sm_count, 8);
    if (prec == 1) return launch_chained(k_init<float>, g, 256, 0, s, 8 * N, kChainBytes, static_cast<float2 *>(psi), N, idx);
    return launch_chained(k_init<double>, g, 256, 0, s, 16 * N, kChainBytes, static_cast<double2 *>(psi), N, idx);
}

// the resident blocks of the sums (256 threads of at most 48 registers)
int reduce_blocks(int sm_count) { return sm_count * 5; }

// Blocks of a pass over n amplitudes, `per` to a block and iteration.
static int sum_blocks(uint64_t n, uint64_t per, int nb) {
    const uint64_t need = (n + per - 1) / per;
    return (int)(need < (uint64_t)nb ? (need < 1 ? 1 : need) : (uint64_t)nb);
}

template <typename T>
static cudaError_t digit_norms_t(const v2<T> *psi, uint64_t N, uint64_t s, int d, double *part, int nb,
                                 double *out_dev, cudaStream_t st) {
    const uint64_t P = s * (uint64_t)d, per = (uint64_t)kSumGroup<T> * kRedBlock;
    int blocks;
    if (d == 1) {
        blocks = sum_blocks(N, per, nb);
        k_norm_partial<T><<<blocks, kRedBlock, 0, st>>>(psi, N, part);
    } else if (P <= kPeriodMax && d <= kPeriodDim) {
        // up to this period the walk needs no index arithmetic at all, and the
        // threads lost to the rounding of A are at most 1 in 11 of a full grid
        blocks = sum_blocks(N, per, nb);
        const int least = (int)((P + kRedBlock - 1) / kRedBlock);
        blocks = blocks < least ? least : blocks;
        const uint32_t A = (uint32_t)((uint64_t)blocks * kRedBlock / P * P);
        k_digit_partial<T><<<blocks, kRedBlock, 0, st>>>(psi, N, (uint32_t)s, (uint32_t)d, A, part);
    } else {
        const uint64_t M = N / (uint64_t)d;
        blocks = sum_blocks(M, per, nb);
        if (s >= per) k_slice_partial<T, true><<<dim3(blocks, d), kRedBlock, 0, st>>>(psi, M, make_fastdiv64(s), P, part);
        else k_slice_partial<T, false><<<dim3(blocks, d), kRedBlock, 0, st>>>(psi, M, make_fastdiv64(s), P, part);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_sum_partials<<<d, 256, 0, st>>>(part, blocks, out_dev);
    return cudaGetLastError();
}

cudaError_t digit_norms(const void *psi, int prec, uint64_t N, uint64_t s, int d, double *part, int nb,
                        double *out_dev, cudaStream_t st) {
    if (prec == 1) return digit_norms_t<float>(static_cast<const float2 *>(psi), N, s, d, part, nb, out_dev, st);
    return digit_norms_t<double>(static_cast<const double2 *>(psi), N, s, d, part, nb, out_dev, st);
}

cudaError_t probabilities(const void *psi, int prec, uint64_t N, double *out, int sm_count, cudaStream_t s) {
    const bool pairs = reinterpret_cast<uintptr_t>(out) % 16 == 0;
    const int g = grid_for(N, pairs ? 4 * kRedBlock : kRedBlock, sm_count, 8);
    if (prec == 1) {
        if (pairs) k_probs<float, true><<<g, kRedBlock, 0, s>>>(static_cast<const float2 *>(psi), N, out);
        else k_probs<float, false><<<g, kRedBlock, 0, s>>>(static_cast<const float2 *>(psi), N, out);
    } else {
        if (pairs) k_probs<double, true><<<g, kRedBlock, 0, s>>>(static_cast<const double2 *>(psi), N, out);
        else k_probs<double, false><<<g, kRedBlock, 0, s>>>(static_cast<const double2 *>(psi), N, out);
    }
    return cudaGetLastError();
}

cudaError_t overlap(const void *a, int prec_a, const void *b, int prec_b, uint64_t N, double *part, int nb,
                    double *out_dev, cudaStream_t s) {
    nb = sum_blocks(N, 4 * kRedBlock, nb);
    if (prec_a == 1 && prec_b == 1)
        k_overlap_partial<float, float><<<nb, kRedBlock, 0, s>>>(static_cast<const float2 *>(a), static_cast<const float2 *>(b), N, part);
    else if (prec_a == 1)
        k_overlap_partial<float, double><<<nb, kRedBlock, 0, s>>>(static_cast<const float2 *>(a), static_cast<const double2 *>(b), N, part);
    else if (prec_b == 1)
        k_overlap_partial<double, float><<<nb, kRedBlock, 0, s>>>(static_cast<const double2 *>(a), static_cast<const float2 *>(b), N, part);
    else
        k_overlap_partial<double, double><<<nb, kRedBlock, 0, s>>>(static_cast<const double2 *>(a), static_cast<const double2 *>(b), N, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_sum_pairs<<<1, 256, 0, s>>>(part, nb, out_dev);
    return cudaGetLastError();
}

uint64_t cdf_chunks(uint64_t N) { return (N + kChunk - 1) / kChunk; }

cudaError_t cdf(const void *psi, int prec, uint64_t N, double *chunk_sums, double *out, cudaStream_t s) {
    const uint64_t nb = cdf_chunks(N);
    if (nb > 0x7fffffffull) return cudaErrorInvalidValue;
    // a caller's complex64 state (qd_cdf_noalloc) may be only 8-byte aligned
    if (prec == 1 && reinterpret_cast<uintptr_t>(psi) % 16 == 0)
        k_chunk_sums<float, true><<<(unsigned)nb, kScanBlock, 0, s>>>(static_cast<const float2 *>(psi), N, chunk_sums);
    else if (prec == 1)
        k_chunk_sums<float, false><<<(unsigned)nb, kScanBlock, 0, s>>>(static_cast<const float2 *>(psi), N, chunk_sums);
    else k_chunk_sums<double, true><<<(unsigned)nb, kScanBlock, 0, s>>>(static_cast<const double2 *>(psi), N, chunk_sums);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_scan_sums<<<1, 1024, 0, s>>>(chunk_sums, nb);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (prec == 1) k_chunk_scan<float><<<(unsigned)nb, kScanBlock, 0, s>>>(static_cast<const float2 *>(psi), N, chunk_sums, out);
    else k_chunk_scan<double><<<(unsigned)nb, kScanBlock, 0, s>>>(static_cast<const double2 *>(psi), N, chunk_sums, out);
    return cudaGetLastError();
}

uint64_t sample_doubles(uint64_t N) {
    const uint64_t nch = (N + kSampChunk - 1) / kSampChunk, nsup = (nch + kSampSuper - 1) / kSampSuper;
    return nch * kSampBlock + nch + nsup;
}

template <typename T>
static cudaError_t sample_t(const v2<T> *psi, uint64_t N, double *scratch, const double *u_dev, uint64_t seed,
                            int64_t shots, int64_t *out_dev, int sm_count, cudaStream_t s) {
    const uint64_t nch = (N + kSampChunk - 1) / kSampChunk, nsup = (nch + kSampSuper - 1) / kSampSuper;
    if (nch > 0x7fffffffull) return cudaErrorInvalidValue;
    double *pre = scratch, *tot = pre + nch * kSampBlock, *sup = tot + nch;
    constexpr int smem = kSampBlock * kSampRow<T>;
    cudaError_t e = cudaFuncSetAttribute((const void *)k_samp_prefix<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_samp_prefix<T><<<(unsigned)nch, kSampBlock, smem, s>>>(psi, N, pre, tot);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_samp_super<<<(unsigned)nsup, kSampSuper, 0, s>>>(tot, nch, sup);
    if (nsup > 1) k_samp_top<<<1, kSampSuper, 0, s>>>(sup, nsup);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int g = grid_for((uint64_t)shots, 256, sm_count, 4);
    k_samp_draw<T><<<g, 256, 0, s>>>(psi, N, pre, tot, nch, sup, nsup, u_dev, seed, shots, out_dev);
    return cudaGetLastError();
}

cudaError_t sample(const void *psi, int prec, uint64_t N, double *scratch, const double *u_dev, uint64_t seed,
                   int64_t shots, int64_t *out_dev, int sm_count, cudaStream_t s) {
    if (shots <= 0) return cudaSuccess;
    if (prec == 1)
        return sample_t<float>(static_cast<const float2 *>(psi), N, scratch, u_dev, seed, shots, out_dev, sm_count, s);
    return sample_t<double>(static_cast<const double2 *>(psi), N, scratch, u_dev, seed, shots, out_dev, sm_count, s);
}

}  // namespace qd
