// Initialisation and FP64 readout launchers (qd_reduce.cu).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "qd_common.cuh"

namespace qd {

// psi = |idx> : zero every amplitude, set psi[idx] = 1.  prec: 1 = c64, 2 = c128.
cudaError_t init_basis(void *psi, int prec, uint64_t N, uint64_t idx, int sm_count, cudaStream_t s);

// Largest number of partial-sum blocks the sums use per digit (part must hold
// d * reduce_blocks(sm_count) doubles).
int reduce_blocks(int sm_count);

// out_dev[x] = sum of |psi_i|^2 (FP64) over the i whose digit (i / s) mod d is
// x, for x < d; d == 1 gives the squared norm.
cudaError_t digit_norms(const void *psi, int prec, uint64_t N, uint64_t s, int d, double *part, int nb,
                        double *out_dev, cudaStream_t st);

// out_dev[0..1] = <a|b> = sum conj(a_i) b_i (FP64), for states of equal length
// (precisions may differ).  part holds 2 * nb doubles.
cudaError_t overlap(const void *a, int prec_a, const void *b, int prec_b, uint64_t N, double *part, int nb,
                    double *out_dev, cudaStream_t s);

// p[i] = |psi_i|^2 (FP64).
cudaError_t probabilities(const void *psi, int prec, uint64_t N, double *out, int sm_count, cudaStream_t s);

// Inclusive prefix sums of |psi_i|^2 (FP64).  chunk_sums must hold
// cdf_chunks(N) + 1 doubles; on return chunk_sums[cdf_chunks(N)] is the total.
uint64_t cdf_chunks(uint64_t N);
cudaError_t cdf(const void *psi, int prec, uint64_t N, double *chunk_sums, double *out, cudaStream_t s);

// out[s] = smallest i with CDF_i > u_s CDF_{N-1}; u_s from u_dev, or from
// Philox4x64-10 (counter (s,0,0,0), key (seed,0)) when u_dev is null.  psi is
// 16-byte aligned; scratch holds sample_doubles(N) doubles.
uint64_t sample_doubles(uint64_t N);
cudaError_t sample(const void *psi, int prec, uint64_t N, double *scratch, const double *u_dev, uint64_t seed,
                   int64_t shots, int64_t *out_dev, int sm_count, cudaStream_t s);

}  // namespace qd
