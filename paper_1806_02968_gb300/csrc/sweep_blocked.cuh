// Gauss-Seidel sweeps of Alg. 3 on a sparse M by blocks of consecutive rows, for deep level
// schedules (the declarations shared by the solvers and the builder).
#pragma once
#include "sparse.cuh"

namespace lsq {

// State of the one-column CSR solve on the device (pcg_sparse.cu).
struct SpState {
    double rho, hn, gstart, rec;
    int32_t iters, done, status, napply;   // napply: preconditioner applications so far
    unsigned err, pad, r0, r1;
};

constexpr int SB_ROWS = 128;               // rows of an inverted diagonal block

// One sweep over K columns (vectors row-major n x K).
struct SbArgs {
    int64_t n;
    int K;
    const int64_t* mptr;
    const int32_t* mcol;
    const void* mval;          // float or double (the operator's type)
    const int64_t* mdiag;
    const double* mval64;      // FP64 values (the diagonal)
    const void* inv;           // inverses of the lower diagonal blocks
    int inv64;                 // they are doubles; else float pairs (double-float sums only)
    const int32_t* done;       // nothing to do once set
    unsigned* err;
    unsigned max_polls;
    const double* r;           // right-hand side (FP64)
    const double* e_old;       // previous sweep's vector or NULL
    double* e_new;             // every slot SB_EMPTY on entry
    double* out64;             // FP64 copy of e_new, or NULL
    int identity;              // the backward sweep right after one forward sweep from zero
    // convergence check ahead of the sweep (one-column solve), or S = NULL
    SpState* S;
    const double* part;
    int nparts;
    double tol, inner_tol;
    int32_t maxit;
};

// True where sweeps over K columns are expected to take less time by blocks than by rows.
bool sb_pays(const SparseHandle* S, int64_t n, int K, bool m32);
// True when sweeps over K columns of this handle run by blocks.
inline bool sb_use(const SparseHandle* S, int64_t n, int K, bool m32) {
    return S->inv != nullptr && sb_pays(S, n, K, m32);
}
// One sweep in the arithmetic of the operator type: FP32 M with pairs = true in double-float
// (vectors hold pairs), otherwise FP64 sums.  The caller has filled e_new with SB_EMPTY.
lsq_status sb_launch(const SbArgs& a, bool fwd, bool m32, bool pairs, cudaStream_t st);
// The inverted diagonal blocks of a handle whose M and levels are complete: none where no number of
// columns takes the block form, or where there is no memory for them (the row forms need none).
lsq_status sb_build_inverse(SparseHandle* S, int64_t n, bool m32, cudaStream_t st);
// lev1[j] = level + 1 of every row for the forward (lev1_f) and backward (lev1_b) dependencies,
// both zero on entry; *max_f, *max_b the deepest levels.  By blocks, both directions at once.
lsq_status sb_levels(const SparseHandle* S, int64_t n, int* lev1_f, int* lev1_b, int* max_f, int* max_b,
                     unsigned* err, cudaStream_t st);

}  // namespace lsq
