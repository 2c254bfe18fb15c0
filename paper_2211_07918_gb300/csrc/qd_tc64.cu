// Dense gates and fused blocks of complex128 states on the tensor cores.
//
// The FP64 pipe gives 1.25 TFLOP/s: a dense gate of D states takes 4 D FP64
// multiply-adds per amplitude, 6.4 D ps, against the 4.7 ps that reading and
// writing the amplitude takes at the copy rate; from D = 2 on the kernel of
// qd_apply.cuh is bound by it (D = 3: 1.3 TB/s, D = 9: 0.46 TB/s).  Here the
// products run on tcgen05 as exact integers (the error-free splitting of
// Ozaki, Ogita, Oishi and Rump, 2012): every group of D amplitudes and every
// matrix row is scaled by a power of two and cut into seven 8-bit digits,
//     x = 2^e sum_s k_s 2^-(8s-1),   |k_s| <= 128,  s = 1..7,
// 55 fraction bits: the group's largest part keeps every bit and no part is off
// by more than an eighth of a unit of the largest part's last place.  Digits are FP16
// operands (exact), the digit products of equal significance s + t = l share
// an FP32 accumulator in TMEM, whose integer sum stays below 2^23, and the
// eight accumulators l = 2..9 are joined in 64-bit integers and rounded once
// to FP64, ties to even.  Dropped are products below 2^-64 of the scale.  Replayed
// in extended precision on random states and Haar matrices, a gate's error is
// 0.6 (D = 2) to 0.3 (D = 32) of that of the FP64 multiply-adds, which round
// 4 D times.
//
// These errors are relative to the largest member on the scale, while a sum of
// rounded products is off relative to its own terms: an output that takes only
// small members, or a large one by a small entry, would lose the digits below
// 2^-55 of the scale.  So members that the matrix does not couple never share
// one: a matrix that falls into parts (a controlled gate or a gate on one of
// its qudits, as a block; tc_couples) has a scale for each part of each group
// (PARTS), and matrices whose rows share some of their members, or hold
// entries more than 2^12 apart, stay on the FP64 pipe.  With a single scale,
// the half of diag(R, R) at 1e-12 of the other was off by 1e-6 of itself; with
// two by 4e-16.
//
// A tile is 128 rows of 8 NP amplitude slots (K = 16 NP): one group of D
// amplitudes per row, spread evenly over its 2 NP threads, or for D <= 4
// several groups side by side with a block-diagonal matrix.  The matrix digits
// are stacked along N, and the accumulators of consecutive l lie side by side
// in TMEM, so that digit s of the amplitudes meets all its partners in one MMA
// per K step (7 instead of 34; an MMA of up to N = 64 costs the same 50 cycles
// as one of N = 16).  A thread carries at most 4 amplitudes through the whole
// tile: loads them, takes their digits into shared memory, and after the MMAs
// joins and stores the same amplitudes' results.  No warp roles: 4 / NP CTAs
// share an SM (1,024 threads, the TMEM is full) and overlap each other's MMA
// waits, and the next tile's loads are issued before the wait.  What bounds it
// is instruction issue and the ALU pipe (60% busy; 230 instructions per
// amplitude, the digits' shifts and masks and the results' normalisation
// first); the FP64 pipe converts one of an amplitude's two parts, the integer
// units the other.  Above D = 16 one CTA fills an SM and its MMAs (2.5 us a
// tile at D = 32) are not overlapped.
//
// Measured on 3.4e7 amplitudes (1.07 GB read and written), CUDA cores -> here:
// D = 2 530 -> 273 us, D = 3 785 -> 277, D = 4 1043 -> 272 (3.95 TB/s), D = 6
// 1561 -> 337, D = 9 2349 -> 413, D = 27 about 6900 -> 520; D = 9 with a
// diagonal run 4403 -> 554; 4,608 amplitudes at D = 9: 25.2 -> 5.8 us, at
// D = 32: 304 -> 14 us (one thread's serial chain of FP64 operations before).
// Matrices of parts (a gate on the lower qudit; controlled), single scale ->
// a scale per part (the loop over a part's members, uniform in a warp, and up
// to two scales per amplitude): D = 4 278 -> 314 for both (471 with a group per
// row instead of four; CUDA cores 1039), D = 9 413 -> 464; 461 (2321), D = 16
// 356 -> 412; 415 (4113), D = 27 473 -> 526; 524 (8365; 618 for the first with a
// loop for every member).
// 64-bit indices, on the FP64 pipe -> here: D = 3 on 2.6e9 amplitudes 58.9 ->
// 22.0 ms, D = 9 on 2.4e9 163 -> 40, D = 27 586 -> 40 (the kernels hold their
// bases in twice the registers and spill up to 122 bytes).
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

constexpr int kRows = 128;     // rows of a tile (MMA M)
constexpr int kDig = 7;        // digits per number
constexpr int kLev = 8;        // accumulators: digit products of significance l = 2..9
constexpr int kSlots = 4;      // amplitude slots of a thread (one 16-byte piece of each digit's row)

// Exponent fields (FP64 bias) of a group's largest part for which the scaled
// integers and the result stay in the normal range; rows with other groups
// (infinities, NaN, extremely small or large amplitudes) are computed in FP64.
constexpr int kRowExLow = 400, kRowExHigh = 1900;
// ... and of a matrix row's largest entry (checked on the host).
constexpr int kMatExLow = 923, kMatExHigh = 1123;
// ... and how far below it the row's smallest non-zero entry may lie.
constexpr int kMatSpread = 12;

template <typename I>
struct Tc64Args {
    double2 *psi;
    I R, base;
    ExpandT<I> ex;
    int32_t D;   // states of a group
    int32_t ra;  // amplitudes of a thread when a row holds one group: member j is slot j % ra of thread j / ra
    int32_t *err;
    uint32_t *queue;  // [0] tiles handed out beyond the first of each CTA, [1] CTAs that are done
    I off[kMaxD];
    double2 U[kMaxD * kMaxD];  // row-major D x D
};

// A diagonal run's table behind the gate: output j of the group at base b is
// multiplied by T[(b / s_qa + off_j / s_qa + carry) mod TS], as in
// DenseTableArgs.
template <typename I> struct DivOf;
template <> struct DivOf<uint32_t> { using type = FastDiv32; };
template <> struct DivOf<uint64_t> { using type = FastDiv64; };
template <typename I, bool TAB> struct Tc64Tab {};
template <typename I> struct Tc64Tab<I, true> {
    typename DivOf<I>::type divA, divT;
    uint32_t oq[16];
    I thr[16];
    uint32_t carry, tsmask;
    const double2 *tab;
};

// Masks of the members that the matrix mixes, for matrices that fall into
// parts (TcCouples): of input member j with the others of its part, and of the
// members that go into output i.  Every part has a scale of its own.
template <bool PARTS> struct Tc64Parts {};
template <> struct Tc64Parts<true> { uint32_t in[kMaxD], out[kMaxD]; };

// Scale exponent (FP64 bias, of 2^(E - 1022)) of a group or matrix row whose
// largest part has the leading word top: parts are below 1 - 2^-7 of the
// scale, so that the leading field (128 times the part, the bias of 128 and
// 0.502 carried from the biases below) stays below 256.
__device__ __forceinline__ int scale_ex(uint32_t top) { return (int)((top + 0x4000u) >> 20); }

// x scaled by 2^-(E - 1022) in offset binary: digit s is byte 8 - s, biased by
// 128; the addend rounds to nearest at byte 1.
__device__ __forceinline__ uint64_t to_fields(double x, int E) {
    const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
    // the mantissa, its implicit bit at 62 (multiplications: the ALU pipe is the busy one)
    uint64_t v = (uint64_t)l * 1024u + ((uint64_t)(((h & 0xfffffu) | 0x100000u) * 1024u) << 32);
    asm("shr.b64 %0, %1, %2;" : "=l"(v) : "l"(v), "r"(E - (int)((h >> 20) & 0x7ffu)));  // 0 from 64 on
    const int64_t sg = (int64_t)(int32_t)h >> 31;
    // one's complement; half a unit less 1 added, so that ties go down for
    // both signs (parts a quarter of the scale or smaller end in a half often:
    // ties away from zero let the state's norm grow by 5e-18 a gate)
    constexpr uint64_t C = 0x8080808080808080ull - 1;
    return (v ^ (uint64_t)sg) + C;
}

// FP16 pair (digit of a, digit of b) of every byte: 1024 + byte is an FP16
// number by its bits, the bias is subtracted exactly.
__device__ __forceinline__ void to_digits(uint64_t a, uint64_t b, uint32_t *w) {
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
#pragma unroll
    for (int s = 0; s < kDig; ++s) {
        const int byte = 7 - s;  // of the 64-bit number
        uint32_t t = __byte_perm(byte >= 4 ? ah : al, byte >= 4 ? bh : bl, (byte & 3) | ((4 + (byte & 3)) << 8));
        t = (t & 0x00ff00ffu) | 0x64006400u;
        asm("add.rn.f16x2 %0, %1, %2;" : "=r"(w[s]) : "r"(t), "r"(0xe480e480u));  // -1152
    }
}

// One part of a result from its accumulators (exact integers in FP32):
// sum_l acc_l 2^-(8l-2) on the grid 2^-GRID, to be scaled by 2^(e + GRID).
// |sum| < K, so the integer stays below 2^63 with GRID = 63 - ceil(log2 K).
// An accumulator of at most 2^22 is an integer by its bits once 1.5 2^23 is
// added; the offsets are taken off together.
template <int GRID>
__device__ __forceinline__ int64_t sum_levels(const uint32_t *acc, int stride) {
    static_assert(GRID >= 57 && GRID <= 59, "shifts");
    constexpr float M = 12582912.0f;
    constexpr uint32_t MB = 0x4b400000u;
    auto f = [&](int l) { return __uint_as_float(acc[(l - 2) * stride]); };
    // K >= 48: worst-case sums of l = 6 and 7 exceed 2^22 and go through the conversion unit
    auto bits = [&](int l) {
        if (GRID == 57 && l >= 6) return (uint32_t)__float2int_rn(f(l)) + MB;
        return __float_as_uint(f(l) + M);
    };
    constexpr int S2 = GRID - 14;  // shift of l = 2; 8 less for each l
    constexpr float c8 = GRID == 59 ? 0x1p-3f : GRID == 58 ? 0x1p-4f : 0x1p-5f, c9 = c8 * 0x1p-8f;
    constexpr uint64_t off = (uint64_t)MB + ((uint64_t)MB << (S2 - 40)) + ((uint64_t)MB << (S2 - 32)) + ((uint64_t)MB << (S2 - 24)) +
                             ((uint64_t)MB << (S2 - 16)) + ((uint64_t)MB << (S2 - 8)) + ((uint64_t)MB << S2);
    uint64_t y = (uint64_t)0 - off + __float_as_uint(fmaf(f(9), c9, fmaf(f(8), c8, M)));
    y += (uint64_t)bits(7) * (1u << (S2 - 40));
    y += (uint64_t)bits(6) * (1u << (S2 - 32));
    y += (uint64_t)bits(5) * (1u << (S2 - 24));
    y += (uint64_t)bits(4) * (1u << (S2 - 16));
    y += (uint64_t)bits(3) << (S2 - 8);
    y += (uint64_t)(bits(2) << (S2 - 32)) << 32;
    return (int64_t)y;
}

// y 2^e rounded to nearest even, by the integer units.
__device__ __forceinline__ double scaled_int(int64_t y, int e) {
    const int64_t sg = y >> 63;
    uint64_t v = (uint64_t)((y ^ sg) - sg);  // below 2^63
    int z = __clz((int)(uint32_t)(v >> 32));
    if (z == 32) {
        if (v == 0) return 0.0;
        z += __clz((int)(uint32_t)v);
    }
    v <<= z - 1;  // top bit at 62: room for the carry of the rounding
    v += 0x1ffu + ((uint32_t)(v >> 10) & 1u);
    return __longlong_as_double((long long)(((v >> 10) + ((uint64_t)(uint32_t)(e + 63 - z + 1022) << 52)) | ((uint64_t)sg << 63)));
}

// The same by the FP64 pipe: y's halves placed in the mantissas of 2^84 and
// 2^52, the offsets taken off exactly, one rounding in the last addition.
__device__ __forceinline__ double scaled_fp(int64_t y, int e) {
    const double hi = __hiloint2double(0x45300000, (int)((uint32_t)((uint64_t)y >> 32) ^ 0x80000000u));
    const double lo = __hiloint2double(0x43300000, (int)(uint32_t)y);
    const double d = (hi - (0x1p84 + 0x1p63 + 0x1p52)) + lo;
    const int h = __double2hiint(d);
    return __hiloint2double(h + (h ? e << 20 : 0), __double2loint(d));
}

__device__ __forceinline__ void tmem_ld2_nowait(uint32_t taddr, uint32_t *r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr));
}

// Instruction descriptor, kind::f16: FP32 accumulator, FP16 A and B, both K-major.
constexpr uint32_t idesc_f16(uint32_t M, uint32_t N) { return (1u << 4) | ((N >> 3) << 17) | ((M >> 4) << 24); }

template <int NP, int GD> struct Tc64Cfg {
    static constexpr int TPR = 2 * NP;             // threads of a row
    static constexpr int THREADS = kRows * TPR;
    static constexpr int PER_SM = 4 / NP;
    static constexpr int K = 16 * NP;
    static constexpr int GRID = NP == 1 ? 59 : NP == 2 ? 58 : 57;          // result grid: 63 - ceil(log2 K)
    static constexpr uint32_t NCOL = NP == 1 ? 128 : NP == 2 ? 256 : 512;  // TMEM columns, >= kLev * K
    static constexpr uint32_t XB = kRows * K * 2, BB = K * K * 2;          // one digit's operands
    static constexpr uint32_t DATA = kDig * XB + (kDig + 1) * BB;          // the matrix with a slice of zeros
    static constexpr int TG = GD ? kSlots / GD : 1;                        // groups of a thread (GD) or row
    static constexpr int GP = GD ? TPR * TG : 1;                           // groups of a row
    static constexpr int PER_TILE = kRows * GP;
    static_assert(PER_SM * NCOL <= 512 && PER_SM * DATA <= 220 * 1024, "occupancy");
    static_assert(GD == 0 || NP == 1, "several groups share a row of two threads");
};

// Member and group of slot c of a thread; the group's index in the register's
// group order (groups of a row are 128 apart: a warp's loads of one member
// are consecutive).
template <typename I, int NP, int GD> struct Slot {
    using C = Tc64Cfg<NP, GD>;
    static __device__ __forceinline__ int member(int c, int a0) { return GD ? c % (GD ? GD : 1) : a0 + c; }
    static __device__ __forceinline__ I group(I t, int row, int part, int k) {
        return t * (I)C::PER_TILE + (I)((GD ? part * C::TG + k : 0) * kRows + row);
    }
};

// Rows with groups outside the integers' range: the results of one thread's
// amplitudes in FP64, from the (unwritten) state.
template <typename I>
__device__ __forceinline__ double2 entry_of(const Tc64Tab<I, true> &b, I base, int j) {
    const I qb = fdiv(base, b.divA);
    const uint32_t TS = (uint32_t)b.divT.d;
    uint32_t k = b.tsmask ? (uint32_t)qb & b.tsmask : (uint32_t)(qb - fdiv(qb, b.divT) * (I)TS);
    k += b.oq[j] + (b.carry && base - qb * (I)b.divA.d >= b.thr[j] ? 1u : 0u);  // < 2 TS + 1
    if (b.tsmask) k &= b.tsmask;
    else {
        if (k >= TS) k -= TS;
        if (k >= TS) k -= TS;
    }
    return __ldg(b.tab + k);
}
__device__ __forceinline__ double2 times(const double2 u, const double2 v) {
    return make_double2(fma(u.x, v.x, -u.y * v.y), fma(u.x, v.y, u.y * v.x));
}

template <typename I, int NP, int GD>
__device__ __noinline__ void row_in_fp64(const Tc64Args<I> &a, I t, int row, int part, int a0, int na, double2 *o) {
    using S = Slot<I, NP, GD>;
    for (int c = 0; c < na; ++c) {
        const int i = S::member(c, a0);
        const I g = S::group(t, row, part, GD ? c / (GD ? GD : 1) : 0);
        double re = 0.0, im = 0.0;
        if (g < a.R) {
            const I base = expand(g, a.ex) + a.base;
            for (int j = 0; j < a.D; ++j) {
                const double2 u = a.U[i * a.D + j], v = a.psi[base + a.off[j]];
                re = fma(u.x, v.x, re);
                re = fma(-u.y, v.y, re);
                im = fma(u.x, v.y, im);
                im = fma(u.y, v.x, im);
            }
        }
        o[c] = make_double2(re, im);
    }
}

// Digit s of the rows against the matrix digits 1..n stacked along N (chunks of
// at most 256 columns), into the accumulators from block s - 1 on.
template <int NP, int GD, int S1>
__device__ __forceinline__ void issue_digit(uint32_t tmem, uint64_t dx, uint64_t db) {
    using C = Tc64Cfg<NP, GD>;
    constexpr int n = S1 == 1 ? kDig + 1 : (kLev + 1 - S1 < kDig ? kLev + 1 - S1 : kDig);  // s = 1 also clears l = 9
    constexpr int per = 256 / C::K;
#pragma unroll
    for (int j0 = 0; j0 < n; j0 += per) {
        const int m = n - j0 < per ? n - j0 : per;
        const uint32_t idesc = idesc_f16(kRows, (uint32_t)(m * C::K));
#pragma unroll
        for (int ks = 0; ks < NP; ++ks)  // descriptors hold addresses in units of 16 bytes; a K step is 256 bytes
            mma_bf16(tmem + (uint32_t)((S1 - 1 + j0) * C::K), dx + (uint64_t)((S1 - 1) * (C::XB / 16) + ks * 16),
                     db + (uint64_t)(j0 * (C::BB / 16) + ks * 16), idesc, S1 == 1 && ks == 0 ? 0u : 1u);
    }
}

// GD: D when several groups share a row (D = 2, 3, 4), else 0.  TAB: each
// output times its entry of a diagonal run's table (both parts are then
// converted by the integer units: the FP64 pipe has the multiplication).
// With GD, tiles are handed out through a counter: in equal shares the four
// CTAs of an SM, whose warps are not issued evenly, ended at 60 to 100% of the
// launch's time (D = 3: 310 -> 286 us on 3.4e7 amplitudes; with a group per
// row, whose CTAs wait at one more barrier, the shares were better: D = 9 415
// against 485 us).
template <typename I, int NP, int GD, bool TAB, bool PARTS>
__global__ void __launch_bounds__(Tc64Cfg<NP, GD>::THREADS, Tc64Cfg<NP, GD>::PER_SM)
    k_dense_tc64(const __grid_constant__ Tc64Args<I> a, const __grid_constant__ Tc64Tab<I, TAB> tb,
                 const __grid_constant__ Tc64Parts<PARTS> pt) {
    using C = Tc64Cfg<NP, GD>;
    using S = Slot<I, NP, GD>;
    constexpr int TG = C::TG;
    constexpr int GS = GD ? GD : kSlots;  // slots of a group in this thread
    constexpr bool QUEUE = GD != 0;
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *const X = sm, *const B = sm + kDig * C::XB;
    __shared__ uint32_t tmem_base;
    __shared__ __align__(8) uint64_t mbar;
    __shared__ int32_t mat_ex[kMaxD];
    __shared__ uint32_t next_tile[2];
    // largest parts: of a thread's amplitudes, or (PARTS) of each member
    __shared__ uint32_t part_max[GD ? 1 : PARTS ? C::TPR * kSlots : C::TPR][kRows];
    __shared__ int32_t row_odd[PARTS && !GD ? kRows : 1];

    const int tid = threadIdx.x, warp = tid >> 5;
    const int row = tid % kRows, part = tid / kRows;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base)),
                     "r"(C::NCOL)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 32) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    for (uint32_t i = tid; i < C::DATA / 16; i += C::THREADS) reinterpret_cast<uint4 *>(sm)[i] = make_uint4(0, 0, 0, 0);
    if (tid < kMaxD) mat_ex[tid] = 0;
    // one matrix entry per thread.  Read through a generic pointer: as constant
    // operands the lanes' different addresses are served one by one (D = 32:
    // 33 us of a launch)
    static_assert(C::THREADS >= (GD ? GD * GD : 64 * NP * NP), "one matrix entry per thread");
    const double2 *Ug = a.U;
    asm volatile("mov.u64 %0, %0;" : "+l"(Ug));
    const bool mine = tid < a.D * a.D;
    const int mi = mine ? tid / a.D : 0, mj = tid - mi * a.D;
    const double2 u = mine ? Ug[tid] : make_double2(0.0, 0.0);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    chain_release();  // this CTA has its TMEM
    chain_wait();
    // scale of the matrix row (a zero row: any)
    if (mine)
        atomicMax(&mat_ex[mi], (int)max((uint32_t)__double2hiint(u.x) & 0x7fffffffu, (uint32_t)__double2hiint(u.y) & 0x7fffffffu));
    __syncthreads();
    const int mE = mat_ex[mi] ? scale_ex((uint32_t)mat_ex[mi]) : 1023;
    __syncthreads();
    if (mine && mj == 0) mat_ex[mi] = mE;
    // digits of the real embedding, rows 2i: (ur, -ui), 2i + 1: (ui, ur), one block per group of a row
    if (mine) {
        const uint64_t fr = to_fields(u.x, mE), fi = to_fields(u.y, mE), fn = to_fields(-u.y, mE);
        uint32_t w0[kDig], w1[kDig];
        to_digits(fr, fn, w0);
        to_digits(fi, fr, w1);
        for (int gp = 0; gp < C::GP; ++gp) {
            const int first = gp / TG * kSlots + gp % TG * GS;
            const uint32_t so = (uint32_t)(GD ? first + mi : mi / a.ra * kSlots + mi % a.ra);
            const uint32_t si = (uint32_t)(GD ? first + mj : mj / a.ra * kSlots + mj % a.ra);
#pragma unroll
            for (int s = 0; s < kDig; ++s) {
                *reinterpret_cast<uint32_t *>(B + s * C::BB + cm_off(2 * so, 2 * si, C::K)) = w0[s];
                *reinterpret_cast<uint32_t *>(B + s * C::BB + cm_off(2 * so + 1, 2 * si, C::K)) = w1[s];
            }
        }
    }

    const uint32_t tmem = tmem_base;
    const I ntiles = (a.R + C::PER_TILE - 1) / C::PER_TILE;
    const int a0 = part * a.ra;  // first member of this thread (one group per row)
    const int na = GD ? TG * GD : max(0, min(a.ra, a.D - a0));
    I base[TG], nbase[TG];
    double2 v[kSlots];
    auto load = [&](I t, I *b) {
#pragma unroll
        for (int k = 0; k < TG; ++k) {
            const I g = S::group(t, row, part, k);
            const bool in = g < a.R;
            b[k] = in ? expand(g, a.ex) + a.base : 0;
#pragma unroll
            for (int u = 0; u < GS; ++u)
                v[k * GS + u] = in && k * GS + u < na ? a.psi[b[k] + a.off[S::member(k * GS + u, a0)]] : make_double2(0.0, 0.0);
        }
    };

    bool dead = false, issued = false;
    uint32_t par = 0, coming = 0;
    if (QUEUE && tid == 0) coming = gridDim.x + atomicAdd(a.queue, 1u);  // the tile after this one
    I t = (I)blockIdx.x;
    if (t < ntiles) load(t, base);
    while (t < ntiles) {
        int E[PARTS ? kSlots : TG];  // of the inputs
        uint32_t Eo[2] = {};         // PARTS: of the outputs, 16 bits each
        bool odd = false;
        auto top_of = [](const double2 x) {
            return max((uint32_t)__double2hiint(x.x) & 0x7fffffffu, (uint32_t)__double2hiint(x.y) & 0x7fffffffu);
        };
        // 1 (an exponent of 0) for parts whose leading words are zero and others not
        auto tiny_of = [](const double2 x) { return (__double2loint(x.x) | __double2loint(x.y)) != 0 ? 1u : 0u; };
        if constexpr (PARTS && GD) {  // whole groups in this thread
            uint32_t top[kSlots];
#pragma unroll
            for (int c = 0; c < TG * GS; ++c) {
                top[c] = top_of(v[c]);
                top[c] = top[c] ? top[c] : tiny_of(v[c]);
            }
#pragma unroll
            for (int c = 0; c < TG * GS; ++c) {
                uint32_t ti = 0, to = 0;
#pragma unroll
                for (int u = 0; u < GS; ++u) {
                    if (pt.in[c % GS] >> u & 1u) ti = max(ti, top[c / GS * GS + u]);
                    if (pt.out[c % GS] >> u & 1u) to = max(to, top[c / GS * GS + u]);
                }
                E[c] = ti ? scale_ex(ti) : 1023;
                odd = odd || E[c] < kRowExLow || E[c] > kRowExHigh;
                Eo[c / 2] |= (uint32_t)(to ? scale_ex(to) : 1023) << (c % 2 * 16);
            }
        } else if constexpr (PARTS) {
#pragma unroll
            for (int c = 0; c < kSlots; ++c)
                if (c < na) {
                    const uint32_t top = top_of(v[c]);
                    part_max[a0 + c][row] = top ? top : tiny_of(v[c]);
                }
            __syncthreads();
            auto scale_of = [&](uint32_t m) {  // the mask is the same for a warp's lanes
                uint32_t top = 0;
                for (; m; m &= m - 1) top = max(top, part_max[__ffs((int)m) - 1][row]);
                const int e = top ? scale_ex(top) : 1023;
                odd = odd || e < kRowExLow || e > kRowExHigh;
                return e;
            };
#pragma unroll
            for (int c = 0; c < kSlots; ++c) {
                E[c] = 1023;
                if (c < na) {
                    const uint32_t in = pt.in[a0 + c], out = pt.out[a0 + c];
                    // (a gate on the lower qudits of a block: neighbours are of one part)
                    E[c] = c && in == pt.in[a0 + c - (c ? 1 : 0)] ? E[c ? c - 1 : 0] : scale_of(in);
                    Eo[c / 2] |= (uint32_t)(out == in ? E[c] : scale_of(out)) << (c % 2 * 16);
                }
            }
        } else
#pragma unroll
        for (int k = 0; k < TG; ++k) {
            uint32_t top = 0;
#pragma unroll
            for (int u = 0; u < GS; ++u) top = max(top, top_of(v[k * GS + u]));
            // (two forms of the same: each spills registers where the other does not, D = 9 413 -> 455 us)
            if constexpr (NP == 2 && !TAB) {
                uint32_t tiny = 0;
#pragma unroll
                for (int u = 0; u < GS; ++u) tiny |= tiny_of(v[k * GS + u]);
                top = top ? top : tiny;
            } else if (top == 0u) {
#pragma unroll
                for (int u = 0; u < GS; ++u) top |= tiny_of(v[k * GS + u]);
            }
            if constexpr (GD == 0) {
                part_max[part][row] = top;
                __syncthreads();
#pragma unroll
                for (int p = 0; p < C::TPR; ++p) top = max(top, part_max[p][row]);
            }
            E[k] = top ? scale_ex(top) : 1023;
            odd = odd || E[k] < kRowExLow || E[k] > kRowExHigh;
        }
        // digits into shared memory: the previous tile's MMAs have completed
        // (every thread waited for them), so the operands may be overwritten;
        // slots that hold nothing keep their zeros
        if (na > 0) {
            uint32_t w[kSlots][kDig];
#pragma unroll
            for (int c = 0; c < kSlots; ++c) {
                if (c < TG * GS && c < na) {
                    const int e = E[PARTS ? c : c / GS];
                    to_digits(to_fields(v[c].x, e), to_fields(v[c].y, e), w[c]);
                } else {
#pragma unroll
                    for (int s = 0; s < kDig; ++s) w[c][s] = 0u;
                }
            }
            unsigned char *dst = X + cm_off((uint32_t)row, (uint32_t)(2 * part * kSlots), C::K);
#pragma unroll
            for (int s = 0; s < kDig; ++s)
                *reinterpret_cast<uint4 *>(dst + s * C::XB) = make_uint4(w[0][s], w[1][s], w[2][s], w[3][s]);
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        // (two entries: a thread may read this one while thread 0 is a tile ahead)
        if (QUEUE && tid == 0) next_tile[par] = coming;
        bool any_odd = false;
        if (__syncthreads_or(odd || dead)) {  // rare: both reasons told apart by a second vote
            if (__syncthreads_or(dead)) break;
            any_odd = true;
            if constexpr (PARTS && !GD) {  // the whole row, whichever part it was
                if (part == 0) row_odd[row] = 0;
                __syncthreads();
                if (odd) row_odd[row] = 1;
                __syncthreads();
                odd = row_odd[row] != 0;
            }
        }
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint64_t dx = smem_desc(smem_u32(X), 128u, C::K * 16u), db = smem_desc(smem_u32(B), 128u, C::K * 16u);
            issue_digit<NP, GD, 1>(tmem, dx, db);
            issue_digit<NP, GD, 2>(tmem, dx, db);
            issue_digit<NP, GD, 3>(tmem, dx, db);
            issue_digit<NP, GD, 4>(tmem, dx, db);
            issue_digit<NP, GD, 5>(tmem, dx, db);
            issue_digit<NP, GD, 6>(tmem, dx, db);
            issue_digit<NP, GD, 7>(tmem, dx, db);
            mma_commit(smem_u32(&mbar));
        }
        __syncwarp();
        issued = true;
        const I nt = QUEUE ? (I)next_tile[par] : t + (I)gridDim.x;
        if (nt < ntiles) {
            if (QUEUE && tid == 0) coming = gridDim.x + atomicAdd(a.queue, 1u);
            load(nt, nbase);  // in flight during the wait
        }
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
            // an amplitude at a time: its 16 accumulators beside the next tile's
            // loads are what 64 registers hold (two at a time spilled them, and
            // a spilled load is waited for: D = 9 415 -> 481 us)
#pragma unroll
            for (int c = 0; c < TG * GS; ++c) {
                if (c < na) {
                    uint32_t acc[kLev][2];
#pragma unroll
                    for (int l = 0; l < kLev; ++l) tmem_ld2_nowait(lane + (uint32_t)(l * C::K + 2 * c), acc[l]);
                    tmem_wait_ld();
                    const int k = c / GS, j = S::member(c, a0);
                    const int e = (PARTS ? (int)(Eo[c / 2] >> (c % 2 * 16) & 0xffffu) : E[k]) + mat_ex[j] - 2044 - C::GRID;
                    if (S::group(t, row, part, k) < a.R && !odd) {
                        const int64_t yr = sum_levels<C::GRID>(&acc[0][0], 2), yi = sum_levels<C::GRID>(&acc[0][1], 2);
                        if constexpr (TAB)
                            a.psi[base[k] + a.off[j]] = times(entry_of(tb, base[k], j), make_double2(scaled_int(yr, e), scaled_int(yi, e)));
                        else
                            a.psi[base[k] + a.off[j]] = make_double2(scaled_fp(yr, e), scaled_int(yi, e));
                    }
                }
            }
        }
        if (any_odd) {  // uniform: these rows were left unwritten above; all their reads before any write
            double2 o[kSlots];
            if (odd) row_in_fp64<I, NP, GD>(a, t, row, part, a0, na, o);
            __syncthreads();
            if (odd && !dead)
                for (int c = 0; c < na; ++c) {
                    const I g = S::group(t, row, part, GD ? c / GS : 0);
                    if (g >= a.R) continue;
                    const I b = expand(g, a.ex) + a.base;
                    if constexpr (TAB) o[c] = times(entry_of(tb, b, S::member(c, a0)), o[c]);
                    a.psi[b + a.off[S::member(c, a0)]] = o[c];
                }
        }
#pragma unroll
        for (int k = 0; k < TG; ++k) base[k] = nbase[k];
        t = nt;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    // the last CTA leaves the queue as it found it, for the register's next launch
    if (QUEUE && tid == 0) __threadfence();
    if (QUEUE && tid == 0 && atomicAdd(a.queue + 1, 1u) == gridDim.x - 1) {
        a.queue[0] = 0;
        a.queue[1] = 0;
    }
    if (warp == 0) {
        if (dead && issued)  // the MMAs in flight read shared memory and write TMEM: a last bounded wait
            for (uint32_t it = 0; it < kWaitLimit; ++it)
                if (mbar_try(smem_u32(&mbar), par ^ 1u)) break;
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(C::NCOL) : "memory");
    }
}

template <typename I, int NP, int GD, bool TAB, bool PARTS>
cudaError_t launch_tab(const GatePlan &g, const TcCouples &tc, void *psi, int sm_count, int32_t *err, cudaStream_t s) {
    using C = Tc64Cfg<NP, GD>;
    Tc64Args<I> a;
    a.psi = static_cast<double2 *>(psi);
    a.R = (I)g.R;
    a.base = (I)g.base_off;
    if constexpr (sizeof(I) == 4) a.ex = narrow(g.ex);
    else a.ex = g.ex;
    a.D = g.D;
    a.ra = GD ? kSlots : (g.D + C::TPR - 1) / C::TPR;
    a.err = err;
    a.queue = reinterpret_cast<uint32_t *>(err) + 2;
    Tc64Tab<I, TAB> tb;
    if constexpr (TAB) {
        if constexpr (sizeof(I) == 4) {
            tb.divA = make_fastdiv32((uint32_t)g.tab_div);
            tb.divT = make_fastdiv32((uint32_t)g.tab_size);
        } else {
            tb.divA = make_fastdiv64(g.tab_div);
            tb.divT = make_fastdiv64(g.tab_size);
        }
        tb.carry = 0;
        for (int j = 0; j < 16; ++j) {
            const uint64_t o = j < g.D ? (uint64_t)g.off[j] : 0;
            tb.oq[j] = (uint32_t)((o / g.tab_div) % g.tab_size);
            tb.thr[j] = (I)(g.tab_div - o % g.tab_div);
            if (o % g.tab_div) tb.carry = 1;
        }
        tb.tsmask = (g.tab_size & (g.tab_size - 1)) == 0 ? (uint32_t)(g.tab_size - 1) : 0u;
        tb.tab = static_cast<const double2 *>(g.tab);
    }
    for (int j = 0; j < kMaxD; ++j) a.off[j] = j < g.D ? (I)g.off[j] : 0;
    for (int k = 0; k < g.D * g.D; ++k) a.U[k] = make_double2(g.U[2 * k], g.U[2 * k + 1]);
    Tc64Parts<PARTS> pt;
    if constexpr (PARTS)
        for (int j = 0; j < kMaxD; ++j) {
            pt.in[j] = j < g.D ? tc.of_col[j] : 0u;
            pt.out[j] = j < g.D ? tc.of_row[j] : 0u;
        }
    auto fn = k_dense_tc64<I, NP, GD, TAB, PARTS>;
    // 4 / NP CTAs on an SM, by their threads and the TMEM; the default split of
    // the L1 memory held one CTA less
    cudaError_t e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::DATA);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    const uint64_t tiles = (g.R + C::PER_TILE - 1) / C::PER_TILE;
    const int grid = (int)std::min<uint64_t>(tiles, (uint64_t)sm_count * C::PER_SM);
    if (grid <= 0) return cudaSuccess;
    // Not chained: launches of about a tile per SM where SMs hold several CTAs.
    // The next launch's CTAs come early, some SMs get several of them and others
    // none, and their tiles take longer than the launch latency that is gained.
    // us per gate, unchained / chained, tiles in brackets, on 152 SMs.  Four CTAs
    // an SM: D = 4 5.8 / 5.5 (64), 5.8 / 7.1 (128), 6.8 / 7.4 (256), 9.9 / 8.0 (512);
    // D = 6 4.9 / 4.4 (64), 4.9 / 6.4 (128), 6.5 / 6.9 (256), 9.2 / 7.4 (512); D = 8
    // 5.3 / 5.3 (64), 5.3 / 7.5 (128), 7.2 / 7.8 (256), 10.5 / 8.7 (512).  Two: D = 16
    // 7.4 / 6.5 (16), 7.3 / 7.6 (32), 7.4 / 8.9 (64), 7.5 / 9.5 (128), 11.1 / 9.8 (256);
    // D = 9 6.0 / 5.4 (52), 8.1 / 6.3 (154).  One: D = 27 13.1 / 11.4 (52).
    const uint64_t sms = (uint64_t)sm_count;
    const bool alone = NP == 1 ? tiles > sms / 2 && tiles <= 2 * sms : NP == 2 ? tiles > sms * 3 / 8 && tiles <= sms : false;
    return launch_chained(fn, grid, C::THREADS, C::DATA, s, 16 * g.N, alone ? 0 : kChainL2Bytes, a, tb, pt);
}

template <typename I, int NP, int GD, bool PARTS>
cudaError_t launch_np(const GatePlan &g, const TcCouples &tc, void *psi, int sm_count, int32_t *err, cudaStream_t s) {
    if constexpr (NP <= 2)
        if (g.tab) return launch_tab<I, NP, GD, true, PARTS>(g, tc, psi, sm_count, err, s);
    return launch_tab<I, NP, GD, false, PARTS>(g, tc, psi, sm_count, err, s);
}

template <typename I, bool PARTS>
cudaError_t launch_rows(const GatePlan &g, const TcCouples &tc, void *psi, int sm_count, int32_t *err, cudaStream_t s) {
    if (g.D <= 8) return launch_np<I, 1, 0, PARTS>(g, tc, psi, sm_count, err, s);
    if (g.D <= 16) return launch_np<I, 2, 0, PARTS>(g, tc, psi, sm_count, err, s);
    if (g.D <= 24) return launch_np<I, 3, 0, PARTS>(g, tc, psi, sm_count, err, s);
    return launch_np<I, 4, 0, PARTS>(g, tc, psi, sm_count, err, s);
}

template <typename I>
cudaError_t launch_i(const GatePlan &g, const TcCouples &tc, void *psi, int sm_count, int32_t *err, cudaStream_t s) {
    if (!tc.one) switch (g.D) {
        case 3: return launch_np<I, 1, 3, true>(g, tc, psi, sm_count, err, s);
        case 4: return launch_np<I, 1, 4, true>(g, tc, psi, sm_count, err, s);
        default: return launch_rows<I, true>(g, tc, psi, sm_count, err, s);
    }
    switch (g.D) {
        case 2: return launch_np<I, 1, 2, false>(g, tc, psi, sm_count, err, s);
        case 3: return launch_np<I, 1, 3, false>(g, tc, psi, sm_count, err, s);
        case 4: return launch_np<I, 1, 4, false>(g, tc, psi, sm_count, err, s);
        default: return launch_rows<I, false>(g, tc, psi, sm_count, err, s);
    }
}

}  // namespace

bool tc_couples(const double *U, int D, int low_top, int high_top, int spread, TcCouples &c) {
    const uint32_t all = D >= 32 ? ~0u : (1u << D) - 1u;
    uint32_t part[kMaxD];
    int n = 0;
    c.one = true;
    for (int j = 0; j < D; ++j) c.of_col[j] = 1u << j;
    for (int i = 0; i < D; ++i) {
        uint32_t m = 0;
        int top = 0, low = 0x7ff;
        for (int j = 0; j < D; ++j) {
            uint64_t p[2];
            std::memcpy(p, &U[2 * (i * D + j)], 16);
            const uint64_t larger = std::max(p[0] & ~(1ull << 63), p[1] & ~(1ull << 63));
            if (!larger) continue;
            const int e = (int)(larger >> 52);
            top = std::max(top, e);
            low = std::min(low, e);
            m |= 1u << j;
        }
        c.of_row[i] = m;
        if (!m) continue;
        if (top < low_top || top > high_top || top - low > spread) return false;
        if (m != all) c.one = false;
        bool known = false;
        for (int k = 0; k < n; ++k) {
            if (part[k] == m) known = true;
            else if (part[k] & m) return false;
        }
        if (known) continue;
        part[n++] = m;
        for (int j = 0; j < D; ++j)
            if (m >> j & 1u) c.of_col[j] = m;
    }
    return true;
}

bool tc64_matrix(const double *U, int D) {
    TcCouples c;
    return tc_couples(U, D, kMatExLow, kMatExHigh, kMatSpread, c);
}

bool tc64_takes(const GatePlan &g, TcCouples &c) {
    if (g.kind != Kind::Dense || g.mode != Mode::Direct || g.D < 2 || g.D > (g.tab ? 16 : kMaxD)) return false;
    // 5 us of setup against a serial chain of 4 D FP64 multiply-adds per thread:
    // D = 2 6.2 against 6.7 us on 262,144 amplitudes, 19.2 against 12.6 on 2^20;
    // D = 3 6.9 against 6.4 on 196,608; from D = 4 on never slower (D = 9
    // 25 against 6.5 us on 4,608 amplitudes)
    const double amps = (double)g.R * g.D;
    if (g.D == 2 && amps < 300000) return false;
    if (g.D == 3 && amps < 180000) return false;
    return tc_couples(g.U.data(), g.D, kMatExLow, kMatExHigh, kMatSpread, c);
}

cudaError_t launch_dense_tc64(const GatePlan &g, const TcCouples &c, void *psi, int sm_count, int32_t *err, cudaStream_t s) {
    if (!wide_index(g)) return launch_i<uint32_t>(g, c, psi, sm_count, err, s);
    return launch_i<uint64_t>(g, c, psi, sm_count, err, s);
}

}  // namespace qd
