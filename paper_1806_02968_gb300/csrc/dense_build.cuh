// Dense preconditioner setup: the sampled normal matrix on the tensor cores and the
// materialised Gauss-Seidel operator (dense_build.cu).
#pragma once
#include "common.cuh"

namespace lsq {

// M (n x n, exactly symmetric, zero diagonals replaced by 1) from the draws idx, p; *n_fixed
// (device) counts the replaced ones.
lsq_status dense_normal_matrix(const lsq_matrix* A, const int32_t* idx, const double* p, const double* inv_d,
                               int64_t s, double* M, unsigned long long* n_fixed, cudaStream_t st);
// The operator of `sweeps` forward and backward sweeps of Alg. 3 on M, n x n row-major.
lsq_status dense_sgs_operator(int64_t n, int sweeps, const double* M, void* op, int op_dtype, cudaStream_t st);

}  // namespace lsq
