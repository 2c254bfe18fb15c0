// Dense gates and fused blocks of complex64 states of 9 to 16 states on the
// tensor cores (larger blocks: qd_tc.cu).
//
// The products run on tcgen05 as exact integers (the error-free splitting of
// Ozaki, Ogita, Oishi and Rump, 2012), as in qd_tc64.cu: every group of D
// amplitudes and the matrix are scaled by a power of two and cut into
// 9-bit digits, x = 2^e sum_s k_s 2^-(9s-1) with |k_s| <= 256, three of them
// for the state (27 bits: 1/4 of the last place of the group's largest part)
// and four for the matrix, which has one scale (36 bits; a coefficient rounded
// to fewer would act on every group alike, a drift that adds up over a
// circuit).  Digits are FP16 operands (exact); the products of equal
// significance l = s + t = 2..5 share an FP32 accumulator in TMEM, whose
// integer sum stays below 2^24, and the four are joined in FP32 with one
// rounding at the output's last place.  Dropped are products below 2^-35 of
// the scale.
//
// An output's error is thus relative to the largest member of its group (and
// the largest matrix entry), as in the BF16 kernel of qd_tc.cu, whose blocks
// of up to 16 states this one took over.  The CUDA cores' is relative to the
// output's own terms, so of the launches that would run there only those come
// here whose matrix couples all members with entries of like size.  A gate on
// one qudit of a 16-state pair, controlled or not, stays there: 334 against
// 217 us below, but a half at 1e-9 of the other keeps its 24 bits (it became
// zero on a common scale).
//
// A tile is 128 rows of 16 amplitude slots (K = 32), one group of D amplitudes
// per row, spread evenly over its two threads.  The matrix digits are stacked
// along N, so that digit s of the amplitudes meets all its partners in one MMA
// per K step (N = 128, 96, 64).  A thread carries at most 8 amplitudes through
// the whole tile: loads them, takes their digits into shared memory, and after
// the MMAs joins and stores the same amplitudes' results; the next tile's
// loads are issued before the MMA wait, and the four CTAs of an SM (1,024
// threads of 64 registers, 64 KB of loads in flight) overlap each other's
// waits.  It is bound by instruction issue (69 per amplitude, against the 128
// packed multiply-adds with hi and lo coefficients of the CUDA-core kernel).
//
// Measured on 6.7e7 amplitudes (1.07 GB read and written), CUDA cores -> here:
// D = 16 334 -> 217 us (4.95 TB/s), D = 12 303 -> 246 us (6.0e7); D = 9 is a
// tie (178 against 176 us) and stays there, as do 16 consecutive amplitudes
// (330 against 373 us: a thread's eight lie in a line of their own).  Up to
// D = 8 the CUDA cores are not the limit (5.4 to 6.3 TB/s against 4.5 to 5.4),
// above D = 16 the warp-specialised kernel is as fast or faster (D = 18 3.87
// TB/s both, D = 27 4.24 against 3.82).  64-bit indices, CUDA cores -> here:
// D = 10 on 8.8e9 amplitudes 49.1 -> 46.7 ms, D = 13 47.3 -> 41.1, D = 16 (8.5e9)
// 44.2 -> 37.0 (42 bytes spilled).
#include <algorithm>
#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

#include "qd_launch.cuh"
#include "qd_plan.h"
#include "qd_tc.h"
#include "qd_umma.cuh"

namespace qd {

namespace {

constexpr int kRows = 128;  // rows of a tile (MMA M)
constexpr int kMaxDim = 16;
constexpr int kParts = 2;   // threads of a row
constexpr int K = 32;       // reals of a row
constexpr int kXDig = 3;    // digits of an amplitude's part
constexpr int kBDig = 4;    // digits of a matrix entry
constexpr int kLev = 4;     // accumulators: digit products of significance l = 2..5
constexpr int kSlots = 8;   // amplitude slots of a thread (two 16-byte pieces of each digit's row)

// Exponent fields (FP32 bias) of a group's largest part for which the scaled
// numbers and the result stay normal; rows with other groups (infinities, NaN,
// extremely small or large amplitudes) are computed in FP64.
constexpr int kRowExLow = 40, kRowExHigh = 210;
// ... and (FP64 bias) of the matrix' largest entry, and how far below it that
// of a row may lie (checked on the host; 28 bits of the row are left).
constexpr int kMatExLow = 1023 - 20, kMatExHigh = 1023 + 20, kMatRows = 8;
// Single gates and blocks priced on the CUDA cores, which round every product
// to 24 bits of its own: every entry of the matrix must couple (no zeros, a
// row's entries within 2^10), so that no output is small but by cancellation,
// and rows lie within 2^3 of the largest entry (33 bits of each are left;
// a unitary matrix' rows do).
constexpr int kGateRows = 3, kGateSpread = 10;

template <typename I>
struct Tc32Args {
    float2 *psi;
    I R, base;
    ExpandT<I> ex;
    int32_t D;      // states of a group
    int32_t ra;     // amplitudes of a thread: member j is slot j % ra of thread j / ra
    int32_t mat_ex; // exponent field of the matrix' largest part
    int32_t *err;
    I off[kMaxDim];
    double2 U[kMaxDim * kMaxDim];  // row-major D x D
};

// Matrix entry scaled by 2^-(E - 1022) in offset binary: the digits' fields
// are 9 bits from bit 27 up (the leading one 10 bits from bit 54), each biased
// by 256; the addend rounds to nearest at bit 27.
__device__ __forceinline__ uint64_t mat_fields(double x, int E) {
    const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
    const uint32_t mh = (((h << 9) | (l >> 23)) & 0x1fffffffu) | 0x20000000u;
    uint64_t v = ((uint64_t)mh << 32) | (l << 9);
    asm("shr.b64 %0, %1, %2;" : "=l"(v) : "l"(v), "r"(E - (int)((h >> 20) & 0x7ffu)));  // 0 from 64 on
    const int64_t sg = (int64_t)(int32_t)h >> 31;
    constexpr uint64_t C = (1ull << 62) + (1ull << 53) + (1ull << 44) + (1ull << 35) + (1ull << 26) - 1;
    return (v ^ (uint64_t)sg) + C;
}
// FP16 pair (digit of a, digit of b) of a field: 1024 + field is an FP16
// number by its bits, the bias is subtracted exactly.
__device__ __forceinline__ uint32_t mat_digit(uint64_t a, uint64_t b, int s) {
    const int at = 54 - 9 * s;
    uint32_t t = __byte_perm((uint32_t)(a >> at), (uint32_t)(b >> at), 0x5410);
    t = (t & (s == 0 ? 0x03ff03ffu : 0x01ff01ffu)) | 0x64006400u;
    uint32_t w;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(w) : "r"(t), "r"(0xe500e500u));  // -1280
    return w;
}

typedef unsigned long long f2p;
__device__ __forceinline__ f2p pk2(float a, float b) {
    f2p r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ f2p fma2(f2p a, f2p b, f2p c) {
    f2p d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// FP16 pairs (re, im) of an amplitude's three digits.  With M = 1.5 2^23,
// fma(r, 1/q, M) - M is r / q rounded to an integer k, and r - k q is exact
// (the two are within a factor of two, or k = 0).
__device__ __forceinline__ void amp_digits(const float2 v, f2p inv, uint32_t *w) {
    const float M = 12582912.0f;
    const f2p Mp = pk2(M, M), Mn = pk2(-M, -M), one = pk2(1.f, 1.f);
    f2p r = fma2(pk2(v.x, v.y), inv, 0ull);
#pragma unroll
    for (int s = 0; s < kXDig; ++s) {
        const float inv_q = s == 0 ? 256.0f : (s == 1 ? 131072.0f : 67108864.0f);
        const float q = 1.0f / inv_q;
        const f2p k = fma2(fma2(r, pk2(inv_q, inv_q), Mp), one, Mn);
        float kr, ki;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(kr), "=f"(ki) : "l"(k));
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(w[s]) : "f"(ki), "f"(kr));
        if (s + 1 < kXDig) r = fma2(k, pk2(-q, -q), r);
    }
}

// max(top, |re|, |im|), a NaN if one is.
__device__ __forceinline__ float abs_top(float top, const float2 v) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(top), "f"(v.x), "f"(v.y));
    return r;
}

__device__ __forceinline__ void tmem_ld4_nowait(uint32_t taddr, uint32_t *r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

constexpr uint32_t idesc_f16(uint32_t M, uint32_t N) { return (1u << 4) | ((N >> 3) << 17) | ((M >> 4) << 24); }

constexpr int kThreads = kRows * kParts;
constexpr int kPerSm = 4;                                          // CTAs: 1,024 threads, all of the TMEM
constexpr uint32_t kCols = 128;                                    // TMEM columns of a CTA
constexpr uint32_t kXBytes = kRows * K * 2, kBBytes = K * K * 2;   // one digit's operands
constexpr uint32_t kData = kXDig * kXBytes + kBDig * kBBytes;
static_assert(kLev * K <= (int)kCols && kPerSm * kCols <= 512 && kParts * kSlots * 2 == K, "tile");

// Rows with groups outside the range of the digits: the results of one
// thread's amplitudes in FP64, from the (unwritten) state.
template <typename I>
__device__ __noinline__ void row_in_fp64(const Tc32Args<I> &a, I base, int a0, int na, float2 *o) {
    for (int c = 0; c < na; ++c) {
        double re = 0.0, im = 0.0;
        for (int j = 0; j < a.D; ++j) {
            const double2 u = a.U[(a0 + c) * a.D + j];
            const float2 v = a.psi[base + a.off[j]];
            re = fma(u.x, (double)v.x, re);
            re = fma(-u.y, (double)v.y, re);
            im = fma(u.x, (double)v.y, im);
            im = fma(u.y, (double)v.x, im);
        }
        o[c] = make_float2((float)re, (float)im);
    }
}

// Digit S1 of the rows against the matrix digits stacked along N, into the
// accumulators from block S1 - 1 on.
template <int S1>
__device__ __forceinline__ void issue_digit(uint32_t tmem, uint64_t dx, uint64_t db) {
    constexpr int n = kLev + 1 - S1;
    const uint32_t idesc = idesc_f16(kRows, (uint32_t)(n * K));
#pragma unroll
    for (int ks = 0; ks < K / 16; ++ks)  // descriptors hold addresses in units of 16 bytes; a K step is 256 bytes
        mma_bf16(tmem + (uint32_t)((S1 - 1) * K), dx + (uint64_t)((S1 - 1) * (kXBytes / 16) + ks * 16),
                 db + (uint64_t)(ks * 16), idesc, S1 == 1 && ks == 0 ? 0u : 1u);
}

// PAIRS: members 2 i and 2 i + 1 are neighbours at an even index, read and
// written together.
template <typename I, bool PAIRS>
__global__ void __launch_bounds__(kThreads, kPerSm) k_dense_tc32(const __grid_constant__ Tc32Args<I> a) {
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *const X = sm, *const B = sm + kXDig * kXBytes;
    __shared__ uint32_t tmem_base;
    __shared__ __align__(8) uint64_t mbar;
    __shared__ float part_max[kParts][kRows];

    const int tid = threadIdx.x, warp = tid >> 5;
    const int row = tid % kRows, part = tid / kRows;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 32) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    for (uint32_t i = tid; i < kData / 16; i += kThreads) reinterpret_cast<uint4 *>(sm)[i] = make_uint4(0, 0, 0, 0);
    // the matrix through a generic pointer: as constant operands the lanes'
    // different addresses are served one by one
    const double2 *Ug = a.U;
    asm volatile("mov.u64 %0, %0;" : "+l"(Ug));
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    chain_wait();  // (no chain_release(): with it the compiler spilled the prefetched amplitudes, 217 -> 250 us)
    // digits of the real embedding, rows 2i: (ur, -ui), 2i + 1: (ui, ur)
    for (int e = tid; e < a.D * a.D; e += kThreads) {
        const int i = e / a.D, j = e - i * a.D;
        const double2 u = Ug[e];
        const uint64_t fr = mat_fields(u.x, a.mat_ex), fi = mat_fields(u.y, a.mat_ex), fn = mat_fields(-u.y, a.mat_ex);
        const uint32_t so = (uint32_t)(i / a.ra * kSlots + i % a.ra), si = (uint32_t)(j / a.ra * kSlots + j % a.ra);
#pragma unroll
        for (int s = 0; s < kBDig; ++s) {
            *reinterpret_cast<uint32_t *>(B + s * kBBytes + cm_off(2 * so, 2 * si, K)) = mat_digit(fr, fn, s);
            *reinterpret_cast<uint32_t *>(B + s * kBBytes + cm_off(2 * so + 1, 2 * si, K)) = mat_digit(fi, fr, s);
        }
    }

    const uint32_t tmem = tmem_base;
    const I ntiles = (a.R + kRows - 1) / kRows;
    const int a0 = part * a.ra;  // this thread's members are [a0, a0 + na)
    const int na = max(0, min(a.ra, a.D - a0));
    I base = 0, nbase = 0;
    float2 v[kSlots];
    auto load = [&](I t, I &b) {
        const I g = t * kRows + (I)row;
        const bool in = g < a.R;
        b = in ? expand(g, a.ex) + a.base : 0;
        if constexpr (PAIRS) {
#pragma unroll
            for (int c = 0; c < kSlots; c += 2) {
                const float4 q = in && c < na ? *reinterpret_cast<const float4 *>(a.psi + b + a.off[a0 + c])
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
                v[c] = make_float2(q.x, q.y);
                v[c + 1] = make_float2(q.z, q.w);
            }
        } else {
#pragma unroll
            for (int c = 0; c < kSlots; ++c) v[c] = in && c < na ? a.psi[b + a.off[a0 + c]] : make_float2(0.f, 0.f);
        }
    };

    bool dead = false, issued = false;
    uint32_t par = 0;
    I t = (I)blockIdx.x;
    if (t < ntiles) load(t, base);
    for (; t < ntiles; t += (I)gridDim.x) {
        float top = 0.f;
#pragma unroll
        for (int c = 0; c < kSlots; ++c) top = abs_top(top, v[c]);
        part_max[part][row] = top;
        __syncthreads();
        top = abs_top(top, make_float2(part_max[0][row], part_max[1][row]));
        const int E = top != 0.f ? (int)(__float_as_uint(top) >> 23 & 255u) : 127;  // parts are below 2^(E - 126)
        const bool odd = E < kRowExLow || E > kRowExHigh;
        // digits into shared memory: the previous tile's MMAs have completed
        // (every thread waited for them), so the operands may be overwritten;
        // slots that hold nothing keep their zeros
#pragma unroll
        for (int q = 0; q < kSlots / 4; ++q) {
            if (4 * q < na) {
                uint32_t w[4][kXDig];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int c = 4 * q + u;
                    if (c < na) {
                        const float inv = __uint_as_float((uint32_t)(253 - E) << 23);  // 2^-(E - 126)
                        amp_digits(v[c], pk2(inv, inv), w[u]);
                    } else {
#pragma unroll
                        for (int s = 0; s < kXDig; ++s) w[u][s] = 0u;
                    }
                }
                unsigned char *dst = X + cm_off((uint32_t)row, (uint32_t)(2 * (part * kSlots + 4 * q)), K);
#pragma unroll
                for (int s = 0; s < kXDig; ++s)
                    *reinterpret_cast<uint4 *>(dst + s * kXBytes) = make_uint4(w[0][s], w[1][s], w[2][s], w[3][s]);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        bool any_odd = false;
        if (__syncthreads_or(odd || dead)) {  // rare: both reasons told apart by a second vote
            if (__syncthreads_or(dead)) break;
            any_odd = true;
        }
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint64_t dx = smem_desc(smem_u32(X), 128u, K * 16u), db = smem_desc(smem_u32(B), 128u, K * 16u);
            issue_digit<1>(tmem, dx, db);
            issue_digit<2>(tmem, dx, db);
            issue_digit<3>(tmem, dx, db);
            mma_commit(smem_u32(&mbar));
        }
        __syncwarp();
        issued = true;
        const I nt = t + (I)gridDim.x;
        if (nt < ntiles) load(nt, nbase);  // in flight during the wait
        bool ok = false;
        for (uint32_t it = 0; it < kWaitLimit && !ok; ++it) ok = mbar_try(smem_u32(&mbar), par);
        par ^= 1u;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
            dead = true;
            if ((tid & 31) == 0) atomicExch(a.err, 1);
        } else {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t lane = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(2 * part * kSlots);
            const f2p step = pk2(0x1p-9f, 0x1p-9f);
            // 2^(E - 126 - 16) 2^(mat_ex - 1022)
            const float sc = __uint_as_float((uint32_t)(E + a.mat_ex - 1037) << 23);
            const bool put = !odd && t * kRows + (I)row < a.R;
#pragma unroll
            for (int c = 0; c < kSlots; c += 2) {  // two amplitudes at a time
                if (c < na) {
                    uint32_t acc[kLev][4];
#pragma unroll
                    for (int l = 0; l < kLev; ++l) tmem_ld4_nowait(lane + (uint32_t)(l * K + 2 * c), acc[l]);
                    tmem_wait_ld();
                    float2 o[2];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        auto f = [&](int l) { return pk2(__uint_as_float(acc[l][2 * u]), __uint_as_float(acc[l][2 * u + 1])); };
                        const f2p y = fma2(fma2(fma2(fma2(f(3), step, f(2)), step, f(1)), step, f(0)), pk2(sc, sc), 0ull);
                        asm("mov.b64 {%0, %1}, %2;" : "=f"(o[u].x), "=f"(o[u].y) : "l"(y));
                    }
                    if (put) {
                        if constexpr (PAIRS) {
                            *reinterpret_cast<float4 *>(a.psi + base + a.off[a0 + c]) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
                        } else {
                            a.psi[base + a.off[a0 + c]] = o[0];
                            if (c + 1 < na) a.psi[base + a.off[a0 + c + 1]] = o[1];
                        }
                    }
                }
            }
        }
        if (any_odd) {  // uniform: these rows were left unwritten above; all their reads before any write
            const bool mine = odd && !dead && t * kRows + (I)row < a.R;
            float2 o[kSlots];
            if (mine) row_in_fp64<I>(a, base, a0, na, o);
            __syncthreads();
            if (mine)
                for (int c = 0; c < na; ++c) a.psi[base + a.off[a0 + c]] = o[c];
        }
        base = nbase;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        if (dead && issued)  // the MMAs in flight read shared memory and write TMEM: a last bounded wait
            for (uint32_t it = 0; it < kWaitLimit; ++it)
                if (mbar_try(smem_u32(&mbar), par ^ 1u)) break;
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kCols) : "memory");
    }
}

template <typename I, bool PAIRS>
cudaError_t launch_fn(const Tc32Args<I> &a, uint64_t N, int sm_count, cudaStream_t s) {
    auto fn = k_dense_tc32<I, PAIRS>;
    // (the default split of the L1 memory may hold fewer CTAs)
    cudaError_t e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kData);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    const uint64_t tiles = ((uint64_t)a.R + kRows - 1) / kRows;
    const int grid = (int)std::min<uint64_t>(tiles, (uint64_t)sm_count * kPerSm);
    if (grid <= 0) return cudaSuccess;
    return launch_chained(fn, grid, kThreads, kData, s, 8 * N, kChainL2Bytes, a);
}

// Exponent field of the matrix' largest part.
int matrix_top(const GatePlan &g) {
    int top = 0;
    for (int k = 0; k < 2 * g.D * g.D; ++k) {
        uint64_t b;
        std::memcpy(&b, &g.U[k], 8);
        top = std::max(top, (int)((b >> 52) & 0x7ff));
    }
    return top;
}

template <typename I>
cudaError_t launch_i(const GatePlan &g, void *psi, int sm_count, int32_t *err, cudaStream_t s) {
    Tc32Args<I> a;
    a.psi = static_cast<float2 *>(psi);
    a.R = (I)g.R;
    a.base = (I)g.base_off;
    if constexpr (sizeof(I) == 4) a.ex = narrow(g.ex);
    else a.ex = g.ex;
    a.D = g.D;
    a.ra = (g.D + kParts - 1) / kParts;
    a.err = err;
    a.mat_ex = matrix_top(g);
    // the local basis in address order; neighbours at even indices in pairs
    // when the lowest qudit is a target of an even number of levels (then
    // every group base is even) and no pair is split between threads
    int perm[kMaxDim];
    for (int j = 0; j < g.D; ++j) perm[j] = j;
    std::sort(perm, perm + g.D, [&](int x, int y) { return g.off[x] < g.off[y]; });
    bool pairs = g.D % 2 == 0 && g.base_off % 2 == 0 && reinterpret_cast<uintptr_t>(psi) % 16 == 0;
    for (int j = 0; j + 1 < g.D && pairs; j += 2) pairs = g.off[perm[j]] % 2 == 0 && g.off[perm[j + 1]] == g.off[perm[j]] + 1;
    for (int k = 0; k < g.ex.n && pairs; ++k) pairs = g.ex.span[k] % 2 == 0;
    if (pairs && a.ra % 2) ++a.ra;  // at most kSlots: kSlots is even
    for (int j = 0; j < kMaxDim; ++j) a.off[j] = j < g.D ? (I)g.off[perm[j]] : 0;
    for (int i = 0; i < g.D; ++i)
        for (int j = 0; j < g.D; ++j) {
            const double *u = &g.U[2 * (perm[i] * g.D + perm[j])];
            a.U[i * g.D + j] = make_double2(u[0], u[1]);
        }
    return pairs ? launch_fn<I, true>(a, g.N, sm_count, s) : launch_fn<I, false>(a, g.N, sm_count, s);
}

}  // namespace

bool tc_matrix_ordinary(const double *U, int D, int low, int high) {
    for (int i = 0; i < D; ++i) {
        int top = 0;
        for (int k = 0; k < 2 * D; ++k) {
            uint64_t b;
            std::memcpy(&b, &U[2 * i * D + k], 8);
            top = std::max(top, (int)((b >> 52) & 0x7ff));
        }
        if (top && (top < low || top > high)) return false;
    }
    return true;
}

// A single gate leaves the tensor cores where its groups fill one wave of the
// CUDA-core kernel (512 threads an SM, one group each) and more than two tiles
// an SM here.  us per gate, CUDA cores / here, states in L2:
//   groups    32 Ki        64 Ki        76 Ki        80 Ki       112 Ki       160 Ki
//   D = 10  4.73 / 4.59  5.04 / 6.38  5.04 / 6.63  6.78 / 6.94  7.09 / 7.50 10.42 / 9.42
//   D = 12  5.50 / 4.73  5.86 / 6.69  5.89 / 6.88  7.84 / 7.19  7.96 / 7.70 11.95 / 9.90
//   D = 16  6.62 / 5.09  7.14 / 7.35  7.14 / 7.49 10.06 / 7.93 10.26 / 8.53 15.43 / 11.04
// (at D = 10 the second wave, of 256 threads an SM, is the better one too).
bool tc32_takes(const GatePlan &g, bool block, int sm_count) {
    if (g.kind != Kind::Dense || g.mode != Mode::Direct || g.tab || g.D < kTcMinD || g.D > kMaxDim) return false;
    if (!block) {
        if (g.D == kTcMinD || g.cuda_cores) return false;
        const uint64_t sms = (uint64_t)sm_count;
        if (g.R > 256 * sms && g.R <= (g.D == 10 ? 768 : 512) * sms) return false;
        bool consecutive = g.D == kMaxDim;
        for (int j = 0; j < g.D && consecutive; ++j) consecutive = g.off[j] >= 0 && g.off[j] < g.D;
        if (consecutive) return false;
    }
    const int top = matrix_top(g);
    if (top < kMatExLow || top > kMatExHigh) return false;
    if (block) return tc_matrix_ordinary(g.U.data(), g.D, top - kMatRows, top);
    TcCouples c;
    return tc_couples(g.U.data(), g.D, top - kGateRows, top, kGateSpread, c) && c.one;
}

cudaError_t launch_dense_tc32(const GatePlan &g, void *psi, int sm_count, int32_t *err, cudaStream_t s) {
    if (!wide_index(g)) return launch_i<uint32_t>(g, psi, sm_count, err, s);
    return launch_i<uint64_t>(g, psi, sm_count, err, s);
}

}  // namespace qd
