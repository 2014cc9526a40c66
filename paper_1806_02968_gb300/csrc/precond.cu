// Sec. 3.3 (sampled normal matrix) and Alg. 3 (symmetric Gauss-Seidel preconditioner): the
// handle and its C entries.
//
// Dense path (dense_build.cu): M = A_s^T A_s is summed over the draws in a fixed order, exactly
// symmetric, its zero diagonal entries replaced by 1.  The SGS operator of Alg. 3 is then
// materialised: column j of the operator is the result of running the t forward and t
// backward Gauss-Seidel sweeps, in the natural row order, on the unit vector e_j from a
// zero start.  Inside PCG the preconditioner is one parallel matrix-vector product with
// that operator instead of a 2n-step dependency chain per application.
#include "common.cuh"
#include "dense_build.cuh"
#include "sparse.cuh"

#include <algorithm>

namespace lsq {

// The identity operator (t = 0: CG on the column-normalised system, the paper's comparison
// method in Sec. 5)
template <typename OT>
__global__ void k_identity_op(int64_t n, OT* op) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * n; t += (int64_t)gridDim.x * blockDim.x)
        op[t] = (t / n == t % n) ? OT(1) : OT(0);
}

template <typename OT>
__global__ void k_op_apply(int64_t n, int64_t kcols, const OT* op, const double* r, double* z) {
    const int lane = threadIdx.x & 31;
    int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t rowc = warp; rowc < n * kcols; rowc += nw) {
        int64_t c = rowc / n, row = rowc % n;
        const OT* P = op + row * n;
        const double* rc = r + c * n;
        double acc = 0.0;
        for (int64_t l = lane; l < n; l += 32) acc = fma((double)P[l], rc[l], acc);
        acc = warp_sum(acc);
        if (lane == 0) z[c * n + row] = acc;
    }
}

__global__ void k_inv(int64_t n, const double* d, double* dst_d, double* inv_d) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * blockDim.x) {
        double v = d[j];
        dst_d[j] = v;
        inv_d[j] = 1.0 / v;
    }
}

__global__ void k_op_to_f64(int64_t count, const float* src, double* dst) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
         e += (int64_t)gridDim.x * blockDim.x)
        dst[e] = (double)src[e];
}

static lsq_status build_dense(const lsq_matrix* A, const int32_t* idx, const double* p,
                              int64_t s, lsq_precond* H, cudaStream_t st) {
    const int64_t n = A->n;
    Scratch sc;
    LSQ_CUDA(sc.alloc(256, st));
    unsigned long long* n_fixed = sc.as<unsigned long long>();
    LSQ_CUDA(cudaMemsetAsync(n_fixed, 0, 16, st));
    lsq_status r = dense_normal_matrix(A, idx, p, H->inv_d, s, H->M, n_fixed, st);
    if (r != LSQ_OK) return r;
    if (H->sweeps == 0) {   // the comparison method: P = I on the normalised system
        const unsigned gi = (unsigned)std::min<int64_t>((n * n + 255) / 256, 152 * 16);
        if (H->op_dtype == LSQ_F32) k_identity_op<float><<<gi, 256, 0, st>>>(n, (float*)H->op);
        else k_identity_op<double><<<gi, 256, 0, st>>>(n, (double*)H->op);
        count_launch();
    } else {
        r = dense_sgs_operator(n, H->sweeps, H->M, H->op, H->op_dtype, st);
        if (r != LSQ_OK) return r;
    }
    LSQ_CUDA(cudaGetLastError());
    unsigned long long nf = 0;
    LSQ_CUDA(cudaMemcpyAsync(&nf, n_fixed, 8, cudaMemcpyDeviceToHost, st));
    LSQ_CUDA(cudaStreamSynchronize(st));
    H->n_fixed_diag = (int64_t)nf;
    H->nnz_M = n * n;
    H->levels = n;
    return LSQ_OK;
}

static void free_handle(lsq_precond* H) {
    if (!H) return;
    pool_free(H->device, {H->M, H->op, H->colscale, H->inv_d});
    if (H->sp) free_sparse(H->sp, H->device);
    delete H;
}

}  // namespace lsq

using namespace lsq;

extern "C" lsq_status lsq_build_precond(const lsq_matrix* A, const int32_t* idx, const double* p,
                                        const double* colscale, int64_t s, const lsq_opts* o,
                                        lsq_precond** P_out, void* stream) {
    lsq_status st0 = check_matrix(A);
    if (st0 != LSQ_OK) return st0;
    LSQ_CHECK_ARG(o && P_out && idx && p && colscale, "NULL argument");
    LSQ_CHECK_ARG(s > 0, "s must be positive");
    LSQ_CHECK_ARG(o->sweeps >= 0 && o->sweeps <= 64, "sweeps must be in [0, 64]");
    LSQ_CHECK_ARG(o->precond_dtype == LSQ_F64 || o->precond_dtype == LSQ_F32, "precond_dtype must be F64 or F32");
    *P_out = nullptr;
    if (A->dense) LSQ_CHECK_ARG(A->n <= 2048, "dense path supports n <= 2048");
    else LSQ_CHECK_ARG(o->sweeps <= 32, "sparse preconditioners support sweeps <= 32");
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t n = A->n;
    int dev = 0;
    LSQ_CUDA(cudaGetDevice(&dev));
    lsq_precond* H = new lsq_precond();
    H->device = dev;
    H->n = n; H->s = s; H->dense = A->dense ? 1 : 0; H->sweeps = o->sweeps; H->op_dtype = o->precond_dtype;
    auto fail = [&](lsq_status code) { free_handle(H); return code; };
    cudaError_t e;
    if ((e = pool_alloc(&H->colscale, sizeof(double) * n, st)) != cudaSuccess ||
        (e = pool_alloc(&H->inv_d, sizeof(double) * n, st)) != cudaSuccess) {
        set_error(std::string("device memory: ") + cudaGetErrorString(e));
        return fail(LSQ_ERR_NOMEM);
    }
    k_inv<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, colscale, H->colscale, H->inv_d);
    count_launch();
    if (!A->dense) {
        lsq_status rs = build_sparse(A, idx, p, s, H, st);
        if (rs != LSQ_OK) return fail(rs);
        *P_out = H;
        return LSQ_OK;
    }
    if ((e = pool_alloc(&H->M, sizeof(double) * n * n, st)) != cudaSuccess ||
        (e = pool_alloc(&H->op, elem_size(o->precond_dtype) * n * n, st)) != cudaSuccess) {
        set_error(std::string("device memory: ") + cudaGetErrorString(e));
        return fail(LSQ_ERR_NOMEM);
    }
    lsq_status r = build_dense(A, idx, p, s, H, st);
    if (r != LSQ_OK) return fail(r);
    *P_out = H;
    return LSQ_OK;
}

extern "C" void lsq_precond_destroy(lsq_precond* P) { free_handle(P); }

extern "C" lsq_status lsq_precond_get_M(const lsq_precond* P, double* M_out, void* stream) {
    LSQ_CHECK_ARG(P && M_out, "NULL argument");
    LSQ_CHECK_ARG(P->dense, "only dense handles hold a dense M");
    LSQ_CUDA(cudaMemcpyAsync(M_out, P->M, sizeof(double) * P->n * P->n, cudaMemcpyDeviceToDevice,
                             (cudaStream_t)stream));
    LSQ_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    return LSQ_OK;
}

extern "C" lsq_status lsq_precond_get_op(const lsq_precond* P, double* op_out, void* stream) {
    LSQ_CHECK_ARG(P && op_out, "NULL argument");
    LSQ_CHECK_ARG(P->dense, "only dense handles hold a materialised operator");
    cudaStream_t st = (cudaStream_t)stream;
    int64_t cnt = P->n * P->n;
    if (P->op_dtype == LSQ_F64) {
        LSQ_CUDA(cudaMemcpyAsync(op_out, P->op, sizeof(double) * cnt, cudaMemcpyDeviceToDevice, st));
    } else {
        k_op_to_f64<<<(unsigned)std::min<int64_t>((cnt + 255) / 256, 4096), 256, 0, st>>>(cnt, (const float*)P->op, op_out);
        count_launch();
    }
    LSQ_CUDA(cudaGetLastError());
    LSQ_CUDA(cudaStreamSynchronize(st));
    return LSQ_OK;
}

extern "C" lsq_status lsq_precond_get_M_csr(const lsq_precond* P, int64_t* nnz_out, int64_t* row_ptr,
                                            int32_t* col_idx, double* vals, void* stream) {
    LSQ_CHECK_ARG(P && nnz_out, "NULL argument");
    LSQ_CHECK_ARG(!P->dense && P->sp, "only sparse handles hold a CSR M");
    *nnz_out = P->sp->nnz_M;
    cudaStream_t st = (cudaStream_t)stream;
    if (row_ptr) LSQ_CUDA(cudaMemcpyAsync(row_ptr, P->sp->mptr, 8 * (size_t)(P->n + 1), cudaMemcpyDeviceToDevice, st));
    if (col_idx) LSQ_CUDA(cudaMemcpyAsync(col_idx, P->sp->mcol, 4 * (size_t)P->sp->nnz_M, cudaMemcpyDeviceToDevice, st));
    if (vals) LSQ_CUDA(cudaMemcpyAsync(vals, P->sp->mval, 8 * (size_t)P->sp->nnz_M, cudaMemcpyDeviceToDevice, st));
    LSQ_CUDA(cudaStreamSynchronize(st));
    return LSQ_OK;
}

extern "C" lsq_status lsq_precond_apply(const lsq_precond* P, const double* r, double* e,
                                        int64_t k, void* stream) {
    LSQ_CHECK_ARG(P && r && e && k >= 1, "bad argument");
    if (!P->dense) return sparse_apply(P, r, e, k, (cudaStream_t)stream);
    cudaStream_t st = (cudaStream_t)stream;
    unsigned g = (unsigned)std::min<int64_t>((P->n * k * 32 + 255) / 256, 152 * 8);
    if (P->op_dtype == LSQ_F64) k_op_apply<double><<<g, 256, 0, st>>>(P->n, k, (const double*)P->op, r, e);
    else k_op_apply<float><<<g, 256, 0, st>>>(P->n, k, (const float*)P->op, r, e);
    count_launch();
    LSQ_CUDA(cudaGetLastError());
    LSQ_CUDA(cudaStreamSynchronize(st));
    return LSQ_OK;
}
