// Tensor-core fused-block kernel (qd_tc.cu).
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "qd_plan.h"

namespace qd {

// Smallest and largest block dimension the tensor-core kernel is used for.
constexpr int kTcMinD = 9;
constexpr int kTcMaxD = 64;

// Padded dimension of a block: D rounded up to a multiple of 8 (16 above 32).
int tc_padded_dim(int D);
// Bytes of the three BF16 matrix terms of a block with padded dimension Dp.
size_t tc_terms_bytes(int Dp);
// Pack the real embedding of the D x D complex matrix U (interleaved, FP64)
// into three BF16 terms (host), in the kernel's shared-memory layout.
void tc_pack_terms(const double *U, int D, int Dp, uint16_t *out);
int tc_smem_bytes(int Dp);
// Launch one block (g.mode == Mode::Tensor) on a complex64 state.
cudaError_t launch_block_tc(const GatePlan &g, void *psi, int sm_count, int32_t *err, cudaStream_t s);

// Dense gates and blocks of complex64 states of kTcMinD to 16 states
// (qd_tc32.cu): whether the kernel takes a launch (direct geometry, matrix
// entries of ordinary size; for a single gate or a block priced on the CUDA
// cores, the shapes at which it is the faster one), and the launch.
bool tc32_takes(const GatePlan &g, bool block, int sm_count);
cudaError_t launch_dense_tc32(const GatePlan &g, void *psi, int sm_count, int32_t *err, cudaStream_t s);

// Whether the exponent field of every matrix row's largest entry lies in
// [low, high] (rows of zeros aside).
bool tc_matrix_ordinary(const double *U, int D, int low, int high);

// What a dense matrix mixes: row i takes the members of_row[i]; member j
// belongs to the part of_col[j]; one: a single part of all members.
struct TcCouples {
    bool one;
    uint32_t of_row[kMaxD], of_col[kMaxD];
};
// False where the parts are not told apart by the zeros of the rows (two rows
// share some of their members, not all), the exponents of a row's entries
// differ by more than `spread`, or that of its largest part lies outside
// [low_top, high_top].  An output may otherwise be much smaller than the
// largest member of its part for other reasons than cancellation, and a scale
// per part does not hold it to the accuracy of a sum of rounded products.
bool tc_couples(const double *U, int D, int low_top, int high_top, int spread, TcCouples &c);

// Dense gates and blocks of complex128 states (qd_tc64.cu): whether the kernel
// takes a launch (direct geometry, a matrix of full parts with entries of
// ordinary size, for D < 4 enough amplitudes in the gate's slice), with the
// parts, and the launch.  err: the error word, followed by the queue words 2
// and 3, zero between launches; the launches that share it are ordered on one
// stream.
bool tc64_takes(const GatePlan &g, TcCouples &c);
cudaError_t launch_dense_tc64(const GatePlan &g, const TcCouples &c, void *psi, int sm_count, int32_t *err, cudaStream_t s);
// Whether the matrix alone lets a launch be taken.
bool tc64_matrix(const double *U, int D);

}  // namespace qd
