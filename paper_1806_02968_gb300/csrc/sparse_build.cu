// Sec. 3.3 for CSR matrices: the sampled normal matrix M = A_s^T A_s as a CSR SpGEMM, its
// level schedule for the Gauss-Seidel sweeps of Alg. 3, and the transposed pattern of A
// used by the A^T q pass of PCG.
//
// Everything is deterministic: the draws are compacted with integer atomics; the
// transpose of the sampled rows is sorted inside each column; every output entry of the
// SpGEMM sums its candidate products in increasing order of the sampled row.
#include "sweep_blocked.cuh"
#include "values.cuh"

#include <algorithm>
#include <vector>

namespace lsq {

// ---------------------------------------------------------------------------------------
// int64 exclusive scan (three passes, any length)
// ---------------------------------------------------------------------------------------
constexpr int SC_T = 512;
__device__ __forceinline__ int64_t block_excl_scan_i64(int64_t v, int64_t* total) {
    __shared__ int64_t s_w[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int64_t y = lane < nw ? s_w[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int64_t z = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += z;
        }
        if (lane < nw) s_w[lane] = y;
    }
    __syncthreads();
    int64_t off = wid ? s_w[wid - 1] : 0;
    if (total) *total = s_w[nw - 1];
    int64_t r = x - v + off;
    __syncthreads();
    return r;
}
__global__ void k_scan64_tiles(const int64_t* in, int64_t n, int64_t* sums) {
    int64_t i = (int64_t)blockIdx.x * SC_T + threadIdx.x;
    int64_t tot;
    block_excl_scan_i64(i < n ? in[i] : 0, &tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}
__global__ void k_scan64_sums(int64_t* sums, int64_t nt) {
    int64_t carry = 0;
    for (int64_t b = 0; b < nt; b += blockDim.x) {
        int64_t i = b + threadIdx.x, tot;
        int64_t e = block_excl_scan_i64(i < nt ? sums[i] : 0, &tot);
        if (i < nt) sums[i] = e + carry;
        carry += tot;
    }
}
__global__ void k_scan64_apply(const int64_t* in, int64_t n, const int64_t* offs, int64_t* out) {
    int64_t i = (int64_t)blockIdx.x * SC_T + threadIdx.x;
    int64_t tot;
    int64_t e = block_excl_scan_i64(i < n ? in[i] : 0, &tot) + offs[blockIdx.x];
    if (i < n) out[i] = e;
    if (i == n - 1) out[n] = e + in[i];
}
// out[0..n] = exclusive prefix of in[0..n) with out[n] = total; scratch: ceil(n/512) int64
lsq_status scan_i64(const int64_t* in, int64_t n, int64_t* out, int64_t* scratch, cudaStream_t st) {
    if (n == 0) { LSQ_CUDA(cudaMemsetAsync(out, 0, 8, st)); return LSQ_OK; }
    int64_t nt = (n + SC_T - 1) / SC_T;
    k_scan64_tiles<<<(unsigned)nt, SC_T, 0, st>>>(in, n, scratch);
    k_scan64_sums<<<1, 1024, 0, st>>>(scratch, nt);
    k_scan64_apply<<<(unsigned)nt, SC_T, 0, st>>>(in, n, scratch, out);
    count_launch(3);
    LSQ_CUDA(cudaGetLastError());
    return LSQ_OK;
}

// Carves one scratch allocation into 256-byte aligned pieces; the size is computed with
// the same rounding as the carving.
struct Carve {
    size_t sizes[16];
    int n = 0;
    void add(size_t bytes) { sizes[n++] = (bytes + 255) & ~size_t(255); }
    size_t total() const { size_t t = 0; for (int i = 0; i < n; ++i) t += sizes[i]; return t; }
    char* at(char* base, int i) const { size_t o = 0; for (int k = 0; k < i; ++k) o += sizes[k]; return base + o; }
};

static unsigned grid1(int64_t work, int t = 256, int64_t cap = 152 * 32) {
    int64_t g = (work + t - 1) / t;
    return (unsigned)(g < 1 ? 1 : (g > cap ? cap : g));
}

// ---------------------------------------------------------------------------------------
// Draw compaction: count[i] = #draws of row i, prob[i] = p_i
// ---------------------------------------------------------------------------------------
__global__ void k_count_draws(const int32_t* idx, const double* p, int64_t s, int64_t* cnt, double* prob) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < s; t += (int64_t)gridDim.x * blockDim.x) {
        int32_t i = idx[t];
        atomicAdd((unsigned long long*)&cnt[i], 1ull);
        prob[i] = p[t];  // every draw of row i carries the same p_i
    }
}
__global__ void k_flag(const int64_t* cnt, int64_t m, int64_t* flag) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        flag[i] = cnt[i] > 0 ? 1 : 0;
}
// unique rows in increasing order, their scale gamma_u = c_u / (s p_u) and row lengths
__global__ void k_compact(const int64_t* cnt, const double* prob, const int64_t* pos, int64_t m, int64_t s,
                          const int64_t* row_ptr, int32_t* urow, double* gam, int64_t* ulen) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        if (cnt[i] > 0) {
            int64_t u = pos[i];
            urow[u] = (int32_t)i;
            gam[u] = (double)cnt[i] / ((double)s * prob[i]);
            ulen[u] = row_ptr[i + 1] - row_ptr[i];
        }
    }
}
// A_s in CSR: row u holds (j, a_{i_u j} / d_j) for the stored entries of row i_u
template <int DT>
__global__ void k_fill_As(lsq_matrix A, const int32_t* urow, int64_t nu, const int64_t* sptr,
                          const double* inv_d, int32_t* scol, double* sval) {
    const int lane = threadIdx.x & 31;
    int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = warp; u < nu; u += nw) {
        const int64_t i = urow[u];
        const int64_t e0 = A.row_ptr[i], len = A.row_ptr[i + 1] - e0, o = sptr[u];
        for (int64_t k = lane; k < len; k += 32) {
            const int32_t j = A.col_idx[e0 + k];
            scol[o + k] = j;
            sval[o + k] = Val<DT>::load(A.vals, e0 + k) * inv_d[j];
        }
    }
}

// ---------------------------------------------------------------------------------------
// Transpose of a CSR pattern (rows nr, columns nc): the entry count of every column, each
// entry's slot inside its column, then the entries in place and every column sorted by row so
// that the order does not depend on the counting.  tperm[k] = source entry.
// One pass of returning atomics gives the counts and the slots at once; the placed word
// (row << 32 | offset inside the row) is all a column needs to be sorted, and nothing but the
// two outputs is needed as scratch: trow holds the slots (by entry) and tperm the words until
// the sort rewrites both.
// ---------------------------------------------------------------------------------------
__global__ void k_col_slot(const int32_t* col, int64_t nnz, unsigned* ccnt, unsigned* slot) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x)
        slot[e] = atomicAdd(&ccnt[col[e]], 1u);
}
// the counts as int64 (for the scan) and the longest column
__global__ void k_col_len(const unsigned* ccnt, int64_t nc, int64_t* len, int* maxlen) {
    int mx = 0;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += (int64_t)gridDim.x * blockDim.x) {
        const unsigned v = ccnt[c];
        len[c] = (int64_t)v;
        mx = max(mx, (int)v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx > 0) atomicMax(maxlen, mx);
}
// a group of L lanes per row (about the mean row length, a power of two); rows far longer than that are
// set aside for the whole CTA
__global__ void k_col_place(const int64_t* rptr, const int32_t* col, int64_t nr, const int64_t* cptr,
                            const unsigned* slot, unsigned long long* word, int L) {
    __shared__ LongRows s_long;
    const int sub = threadIdx.x & (L - 1);
    const int64_t grp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / L;
    const int64_t ngrp = ((int64_t)gridDim.x * blockDim.x) / L;
    s_long.init();
    for (int64_t r0 = 0; r0 < nr; r0 += ngrp) {   // the same trip count for every group of a warp
        const int64_t r = r0 + grp;
        const int64_t e0 = r < nr ? rptr[r] : 0, e1 = r < nr ? rptr[r + 1] : 0;
        if (s_long.put(sub == 0 && e1 - e0 > LONG_ROW && e1 - e0 > 64 * L, r, L)) continue;
        for (int64_t e = e0 + sub; e < e1; e += L)
            word[cptr[col[e]] + slot[e]] = ((unsigned long long)r << 32) | (unsigned long long)(e - e0);
    }
    s_long.each([&](int64_t r) {
        const int64_t e0 = rptr[r], e1 = rptr[r + 1];
#pragma unroll 4
        for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x)
            word[cptr[col[e]] + slot[e]] = ((unsigned long long)r << 32) | (unsigned long long)(e - e0);
    });
}
constexpr int SPG_CAP = 8192;   // candidate products of one output row

// Ascending bitonic sort of key[0..len) by the threads first, first + nt, ... of one group.  Every
// compare keeps the smaller key at the lower index (the first step of a merge compares
// mirrored positions), so the places from len up to the next power of two act as +infinity
// and are never touched.
template <typename Sync>
__device__ __forceinline__ void bitonic_any(unsigned long long* key, unsigned len, unsigned first, unsigned nt,
                                            Sync sync) {
    unsigned lg = 0;
    while ((1ull << lg) < len) ++lg;
    const unsigned pairs = lg ? 1u << (lg - 1) : 0u;
    auto order = [&](unsigned lo, unsigned hi) {
        if (hi < len) {
            const unsigned long long x = key[lo], y = key[hi];
            if (x > y) { key[lo] = y; key[hi] = x; }
        }
    };
    for (unsigned m = 1; m <= lg; ++m) {          // merges of 2^m keys
        for (unsigned t = first; t < pairs; t += nt) {
            const unsigned o = t & ((1u << (m - 1)) - 1u), base = (t >> (m - 1)) << m;
            order(base + o, base + (1u << m) - 1u - o);
        }
        sync();
        for (int d = (int)m - 2; d >= 0; --d) {   // stride 2^d
            for (unsigned t = first; t < pairs; t += nt) {
                const unsigned lo = ((t >> d) << (d + 1)) + (t & ((1u << d) - 1u));
                order(lo, lo + (1u << d));
            }
            sync();
        }
    }
}
__device__ __forceinline__ void emit_sorted(unsigned long long w, const int64_t* rptr, int32_t* trow, int64_t* tperm) {
    const int64_t r = (int64_t)(w >> 32);
    *trow = (int32_t)r;
    *tperm = rptr[r] + (int64_t)(w & 0xFFFFFFFFull);
}
// Columns of up to CW_CAP entries: a warp per column in its slice of shared memory.  Longer
// ones: a CTA per column, in shared memory of the longest column's size (`cap` words; sized by
// the launch so that short columns leave room for more CTAs), or in place in global memory
// beyond the 8192 words a CTA can hold.
constexpr int CW_CAP = 128;
constexpr int CS_CAP = 8192;
__global__ void __launch_bounds__(256) k_col_sort_warp(const int64_t* cptr, int64_t nc, const int64_t* rptr,
                                                       int32_t* trow, int64_t* tperm) {
    __shared__ unsigned long long s_key[8][CW_CAP];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long* key = s_key[wid];
    const unsigned long long* word = reinterpret_cast<const unsigned long long*>(tperm);
    for (int64_t c = (int64_t)blockIdx.x * 8 + wid; c < nc; c += (int64_t)gridDim.x * 8) {
        const int64_t a = cptr[c], len = cptr[c + 1] - a;
        if (len > CW_CAP || len < 1) continue;
        for (int i = lane; i < len; i += 32) key[i] = word[a + i];
        __syncwarp();
        bitonic_any(key, (unsigned)len, lane, 32u, [] { __syncwarp(); });
        for (int i = lane; i < len; i += 32) emit_sorted(key[i], rptr, trow + a + i, tperm + a + i);
        __syncwarp();
    }
}
__global__ void __launch_bounds__(256) k_col_sort_cta(const int64_t* cptr, int64_t nc, const int64_t* rptr,
                                                      int32_t* trow, int64_t* tperm, int cap) {
    extern __shared__ __align__(16) unsigned long long cs_key[];
    unsigned long long* word = reinterpret_cast<unsigned long long*>(tperm);
    for (int64_t c = blockIdx.x; c < nc; c += gridDim.x) {
        const int64_t a = cptr[c], len = cptr[c + 1] - a;
        if (len <= CW_CAP) continue;
        unsigned long long* key = word + a;
        if (len <= cap) {
            key = cs_key;
            for (int i = threadIdx.x; i < len; i += blockDim.x) key[i] = word[a + i];
            __syncthreads();
        }
        bitonic_any(key, (unsigned)len, threadIdx.x, blockDim.x, [] { __syncthreads(); });
        for (int64_t i = threadIdx.x; i < len; i += blockDim.x) emit_sorted(key[i], rptr, trow + a + i, tperm + a + i);
        __syncthreads();
    }
}

lsq_status transpose_pattern(const int64_t* rptr, const int32_t* col, int64_t nr, int64_t nc, int64_t nnz,
                             int64_t* cptr, int32_t* trow, int64_t* tperm, cudaStream_t st) {
    Scratch sc;
    const int64_t nt = (nc + SC_T - 1) / SC_T + 1;
    LSQ_CUDA(sc.alloc(4 * (size_t)(nc + 4) + 8 * (size_t)(nc + nt + 4), st));
    int64_t* len = sc.as<int64_t>();
    int64_t* ts = len + nc;
    unsigned* ccnt = reinterpret_cast<unsigned*>(ts + nt + 4);   // nc counters, then the longest
    int* maxlen = reinterpret_cast<int*>(ccnt + nc);
    LSQ_CUDA(cudaMemsetAsync(ccnt, 0, 4 * (size_t)(nc + 4), st));
    unsigned* slot = reinterpret_cast<unsigned*>(trow);
    unsigned long long* word = reinterpret_cast<unsigned long long*>(tperm);
    k_col_slot<<<grid1(nnz), 256, 0, st>>>(col, nnz, ccnt, slot);
    k_col_len<<<grid1(nc), 256, 0, st>>>(ccnt, nc, len, maxlen);
    count_launch(2);
    lsq_status s = scan_i64(len, nc, cptr, ts, st);
    if (s != LSQ_OK) return s;
    int hmax = 0;
    LSQ_CUDA(cudaMemcpyAsync(&hmax, maxlen, 4, cudaMemcpyDeviceToHost, st));
    int L = 1;
    while (L < 32 && L * nr < nnz) L <<= 1;
    k_col_place<<<grid1(nr * L), 256, 0, st>>>(rptr, col, nr, cptr, slot, word, L);
    k_col_sort_warp<<<grid1(nc, 8), 256, 0, st>>>(cptr, nc, rptr, trow, tperm);
    count_launch(2);
    LSQ_CUDA(cudaStreamSynchronize(st));   // hmax
    if (hmax > CW_CAP) {
        const int cap = hmax < CS_CAP ? hmax : CS_CAP;
        const int smem = cap * 8;
        LSQ_CUDA(cudaFuncSetAttribute(k_col_sort_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, CS_CAP * 8));
        k_col_sort_cta<<<(unsigned)std::min<int64_t>(nc, 152 * 32), 256, smem, st>>>(cptr, nc, rptr, trow, tperm, cap);
        count_launch();
    }
    LSQ_CUDA(cudaGetLastError());
    return LSQ_OK;
}

// ---------------------------------------------------------------------------------------
// SpGEMM M = A_s^T diag(gamma) A_s, one warp per output row j.  The row's candidates are the
// products (k, gamma_u (a_uj a_uk)) for every sampled row u with an entry in column j (in
// increasing u) and every entry k of that row.
//   Rows of up to SPG_SHORT candidates (a graph's): the candidates wait in shared memory, each
//   finds its column's rank by counting, and the first of a column adds up the others.
//   Longer rows: a bitmap of the n columns (in windows of SPG_WIN) gives the distinct columns in
//   order; a candidate's rank is a prefix of popcounts, and 32 candidates at a time are added to
//   the row's sums in shared memory, candidates of the same column one after the other.
// Either way the sum of a column runs over u in increasing order from 0, so it has the same
// bits however the work is laid out.  Pass 0 counts the distinct columns (the diagonal always
// among them); pass 1 writes the row, 1 / M_jj and the diagonal's position.
// Bound: latency of the gathers of A_s, hidden by as many warps as the bitmap (n / 8 bytes and
// half of that again for the prefixes) and the sums leave room for.
// Sampling and building 4e6 x 40,000 (763 products per row) takes 38.3 ms, against 106.6 ms when
// a CTA sorted a row's candidates in 128 KB of shared memory and one thread added them up
// (58.5 ms) and the transposes sorted every column in 128 KB as well (7.7 ms).
// ---------------------------------------------------------------------------------------
constexpr int SPG_SHORT = 96;
constexpr int64_t SPG_WIN = 1 << 18;   // columns per bitmap window (32 KB, and 16 KB of prefixes)

struct SpgArgs {
    int64_t n;
    const int64_t* sptr;
    const int32_t* scol;
    const double* sval;
    const double* gam;
    const int64_t* tptr;
    const int32_t* trow;
    const int64_t* tperm;
    const int32_t* cand;       // candidates of every row
    int64_t* mcnt;             // pass 0
    int* maxrow;               // pass 0: the longest row
    const int64_t* mptr;       // pass 1
    int32_t* mcol;
    double* mval;
    float* mval32;
    double* dinv;
    int64_t* mdiag;
    unsigned long long* n_fixed;
    int win;                   // columns per window
    int acap;                  // entries of a row's sums
};
// candidates of every row and the largest count
__global__ void k_spg_cand(int64_t n, const int64_t* sptr, const int64_t* tptr, const int32_t* trow, int32_t* cand,
                           int* maxcand) {
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int mx = 0;
    for (int64_t j = w; j < n; j += nw) {
        int64_t t = 0;
        for (int64_t q = tptr[j] + lane; q < tptr[j + 1]; q += 32) {
            const int64_t u = trow[q];
            t += sptr[u + 1] - sptr[u];
        }
        t = warp_sum(t);
        if (t > SPG_CAP) t = SPG_CAP + 1;   // refused by the caller
        if (lane == 0) cand[j] = (int32_t)t;
        mx = max(mx, (int)t);
    }
    if (lane == 0 && mx > 0) atomicMax(maxcand, mx);
}
// Calls fn(column, value, valid) for 32 candidates of row j at a time, in order; the warp runs
// it converged.  With VALS false the values are not formed.
template <bool VALS, typename F>
__device__ __forceinline__ void spg_for_candidates(const SpgArgs& a, int64_t j, int lane, F fn) {
    const int64_t q0 = a.tptr[j], q1 = a.tptr[j + 1];
    for (int64_t qb = q0; qb < q1; qb += 32) {
        const int64_t q = qb + lane;
        int len = 0;
        int64_t e0 = 0;
        double guj = 0.0, auj = 0.0;
        if (q < q1) {
            const int64_t u = a.trow[q];
            e0 = a.sptr[u];
            len = (int)(a.sptr[u + 1] - e0);
            if (VALS) { guj = a.gam[u]; auj = a.sval[a.tperm[q]]; }
        }
        int inc = len;   // inclusive prefix of the lengths
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const int tot = __shfl_sync(0xffffffffu, inc, 31);
        for (int t0 = 0; t0 < tot; t0 += 32) {
            const int t = t0 + lane;
            int src = 0;     // the first lane whose inclusive prefix exceeds t
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const int v = __shfl_sync(0xffffffffu, inc, src + o - 1);
                if (v <= t) src += o;
            }
            src = min(src, 31);
            const int before = __shfl_sync(0xffffffffu, inc - len, src);
            const int64_t base = __shfl_sync(0xffffffffu, e0, src);
            double gu = 0.0, au = 0.0;
            if (VALS) { gu = __shfl_sync(0xffffffffu, guj, src); au = __shfl_sync(0xffffffffu, auj, src); }
            const bool ok = t < tot;
            int32_t k = -1;
            double v = 0.0;
            if (ok) {
                k = a.scol[base + (t - before)];
                if (VALS) v = gu * (au * a.sval[base + (t - before)]);   // M_jk and M_kj get the same bits
            }
            fn(k, v, ok);
        }
    }
}
__device__ __forceinline__ void spg_put(const SpgArgs& a, int64_t j, int64_t at, int32_t k, double v) {
    if ((int64_t)k == j) {
        if (v == 0.0) { v = 1.0; atomicAdd(a.n_fixed, 1ull); }   // never drawn: the diagonal of Â^T Â
        a.dinv[j] = 1.0 / v;
        a.mdiag[j] = at;
    }
    a.mcol[at] = k;
    a.mval[at] = v;
    if (a.mval32) a.mval32[at] = (float)v;
}

constexpr int SPS_W = 4;   // warps per CTA of the short-row kernel
template <bool FILL>
__global__ void __launch_bounds__(32 * SPS_W) k_spgemm_short(SpgArgs a) {
    __shared__ int32_t s_col[SPS_W][SPG_SHORT + 1];
    __shared__ double s_val[SPS_W][FILL ? SPG_SHORT + 1 : 1];
    __shared__ unsigned s_first[SPS_W][(SPG_SHORT + 32) / 32];   // bit i: candidate i is its column's first
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t* col = s_col[wid];
    double* val = s_val[wid];
    unsigned* first = s_first[wid];
    for (int64_t j = (int64_t)blockIdx.x * SPS_W + wid; j < a.n; j += (int64_t)gridDim.x * SPS_W) {
        const int cnt = a.cand[j];
        if (cnt > SPG_SHORT) continue;
        int at = 0;
        spg_for_candidates<FILL>(a, j, lane, [&](int32_t k, double v, bool ok) {
            if (ok) {
                col[at + lane] = k;
                if (FILL) val[at + lane] = v;
            }
            at += __popc(__ballot_sync(0xffffffffu, ok));
        });
        if (lane == 0) {                     // the diagonal, last: adds nothing
            col[cnt] = (int32_t)j;
            if (FILL) val[cnt] = 0.0;
        }
        __syncwarp();
        int uniq = 0;
        for (int b = 0; b <= cnt; b += 32) {
            const int i = b + lane;
            bool f = i <= cnt;
            for (int t = 0; t < min(b + 31, cnt); ++t)
                if (t < i && f && col[t] == col[i]) f = false;
            const unsigned m = __ballot_sync(0xffffffffu, f);
            if (lane == 0) first[b >> 5] = m;
            uniq += __popc(m);
        }
        if (!FILL) {
            if (lane == 0) a.mcnt[j] = uniq;
        } else {
            __syncwarp();
            for (int i = lane; i <= cnt; i += 32) {
                if (!((first[i >> 5] >> (i & 31)) & 1u)) continue;
                const int32_t k = col[i];
                int rank = 0;
                double sum = 0.0;
                for (int t = 0; t <= cnt; ++t) {
                    const int32_t kt = col[t];
                    if (kt == k) sum += val[t];
                    rank += (kt < k && ((first[t >> 5] >> (t & 31)) & 1u)) ? 1 : 0;
                }
                spg_put(a, j, a.mptr[j] + rank, k, sum);
            }
        }
        __syncwarp();
    }
}

template <bool FILL>
__global__ void __launch_bounds__(32) k_spgemm_long(SpgArgs a) {
    extern __shared__ __align__(16) unsigned char spg_smem[];
    const int lane = threadIdx.x;
    // words of the bitmap a lane walks: an odd number, so that the lanes' words lie in distinct banks
    const int words = (a.win + 31) >> 5, per = ((words + 31) >> 5) | 1;
    double* acc = reinterpret_cast<double*>(spg_smem);                       // acap sums (pass 1)
    int32_t* ocol = reinterpret_cast<int32_t*>(acc + (FILL ? a.acap : 0));   // their columns
    unsigned* bits = reinterpret_cast<unsigned*>(ocol + (FILL ? a.acap : 0));
    unsigned short* pre = reinterpret_cast<unsigned short*>(bits + words);   // columns before each word
    int longest = 0;
    for (int64_t j = blockIdx.x; j < a.n; j += gridDim.x) {
        if (a.cand[j] <= SPG_SHORT) continue;
        int64_t out = FILL ? a.mptr[j] : 0;
        int uniq_all = 0;
        for (int64_t w0 = 0; w0 < a.n; w0 += a.win) {
            for (int i = lane; i < words; i += 32) bits[i] = 0u;
            __syncwarp();
            spg_for_candidates<false>(a, j, lane, [&](int32_t k, double, bool ok) {
                const int64_t d = (int64_t)k - w0;
                if (ok && d >= 0 && d < a.win) atomicOr(&bits[d >> 5], 1u << (d & 31));
            });
            if (lane == 0 && j >= w0 && j < w0 + a.win) atomicOr(&bits[(j - w0) >> 5], 1u << ((j - w0) & 31));
            __syncwarp();
            const int i0 = min(lane * per, words), i1 = min(i0 + per, words);
            int mine = 0;
            for (int i = i0; i < i1; ++i) mine += __popc(bits[i]);
            int inc = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            const int uniq = __shfl_sync(0xffffffffu, inc, 31);
            uniq_all += uniq;
            if (FILL) {
                int run = inc - mine;
                for (int i = i0; i < i1; ++i) {
                    pre[i] = (unsigned short)run;
                    unsigned b = bits[i];
                    while (b) {
                        const int t = __ffs(b) - 1;
                        ocol[run++] = (int32_t)(w0 + (int64_t)i * 32 + t);
                        b &= b - 1;
                    }
                }
                for (int i = lane; i < uniq; i += 32) acc[i] = 0.0;
                __syncwarp();
                spg_for_candidates<true>(a, j, lane, [&](int32_t k, double v, bool ok) {
                    const int64_t d = (int64_t)k - w0;
                    const bool in = ok && d >= 0 && d < a.win;
                    // candidates of one column add in order: round r takes each column's r-th lane
                    const unsigned same = __match_any_sync(0xffffffffu, in ? k : -1 - lane);
                    const int my = __popc(same & ((1u << lane) - 1u));
                    int rank = 0;
                    if (in) rank = (int)pre[d >> 5] + __popc(bits[d >> 5] & ((1u << (d & 31)) - 1u));
                    for (int r = 0; __any_sync(0xffffffffu, in && my >= r); ++r) {
                        if (in && my == r) acc[rank] += v;
                        __syncwarp();
                    }
                });
                for (int i = lane; i < uniq; i += 32) spg_put(a, j, out + i, ocol[i], acc[i]);
                out += uniq;
                __syncwarp();
            }
        }
        if (!FILL) {
            if (lane == 0) a.mcnt[j] = uniq_all;
            longest = max(longest, uniq_all);
        }
    }
    if (!FILL && lane == 0 && longest > 0) atomicMax(a.maxrow, longest);
}
// Shared memory of the long-row kernel, and the most any call needs.  The limit that a kernel is
// given is one for the whole process, so it is set to the most: two threads that build handles of
// different sizes must not lower it under one another.
constexpr size_t spg_bytes(bool fill, size_t win, size_t acap) {
    return (fill ? 12 * acap : 0) + 6 * ((win + 31) / 32) + 16;
}
// Both kernels of one pass; the long-row kernel only when there is a long row.
template <bool FILL>
static lsq_status spgemm_pass(SpgArgs a, int maxcand, int sms, cudaStream_t st) {
    k_spgemm_short<FILL><<<(unsigned)std::min<int64_t>((a.n + SPS_W - 1) / SPS_W, (int64_t)sms * 16), 32 * SPS_W, 0, st>>>(a);
    count_launch();
    if (maxcand <= SPG_SHORT) return LSQ_OK;
    a.win = (int)std::min<int64_t>(a.n, SPG_WIN);
    const size_t smem = spg_bytes(FILL, (size_t)a.win, (size_t)a.acap);
    constexpr size_t most = spg_bytes(FILL, (size_t)SPG_WIN, (size_t)SPG_CAP + 2);
    static_assert(most <= 227 * 1024, "a row's sums and the window's bitmap fit an SM");
    LSQ_CUDA(cudaFuncSetAttribute(k_spgemm_long<FILL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
    int per = 0;
    LSQ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_spgemm_long<FILL>, 32, smem));
    if (per < 1) { set_error("SpGEMM kernel does not fit on an SM"); return LSQ_ERR_CUDA; }
    k_spgemm_long<FILL><<<(unsigned)std::min<int64_t>(a.n, (int64_t)sms * per * 2), 32, smem, st>>>(a);
    count_launch();
    return LSQ_OK;
}

// Level schedules: lev_f(j) = 1 + max lev_f(k) over k < j with M_jk != 0 (rows in natural
// order), lev_b(j) = 1 + max lev_b(k) over k > j (reverse order), 0 for a row without such
// entries.  Each schedule lists the rows by level (any order inside a level: those rows are
// independent) with the level of every slot and the number of rows of every level.
//
// k_levels: cooperative launch; warp w takes rows w, w + W, ... in dependency order (natural
// order forward, reverse backward), so every row a row depends on is taken by a warp no later
// than the row itself and, every warp being resident, every wait ends.  lev1 holds level + 1
// (0 = not yet known).  Waits are bounded; one failed wait sets *err and ends them all.
__device__ __forceinline__ int ld_acquire_i32(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_i32(int* p, int v) {
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
template <bool FWD>
__global__ void __launch_bounds__(256) k_levels(int64_t n, const int64_t* mptr, const int32_t* mcol,
                                                const int64_t* mdiag, int* lev1, int* maxlev, unsigned* err,
                                                unsigned max_polls) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t W = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int mymax = 0;
    for (int64_t t = gw; t < n; t += W) {
        const int64_t j = FWD ? t : n - 1 - t;
        const int64_t d0 = FWD ? mptr[j] : mdiag[j] + 1, d1 = FWD ? mdiag[j] : mptr[j + 1];
        int mx = 0;
        // the dependencies in batches of 8 per lane: all loads of a batch are issued
        // together, then only the ones not known yet are polled again
        for (int64_t base = d0 + lane; base < d1; base += 32 * 8) {
            int32_t kk[8];
            int v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) kk[u] = base + 32 * u < d1 ? mcol[base + 32 * u] : -1;
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = kk[u] >= 0 ? ld_acquire_i32(lev1 + kk[u]) : 1;
            unsigned polls = 0, ns = 32;
            while (true) {
                bool missing = false;
#pragma unroll
                for (int u = 0; u < 8; ++u) missing = missing || v[u] == 0;
                if (!missing) break;
                ++polls;
                if (polls > max_polls || ((polls & 255u) == 0 && *(volatile unsigned*)err != 0u)) {
                    atomicOr(err, DEV_ERR_TIMEOUT);
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = max(v[u], 1);
                    break;
                }
                if (polls > 4) { __nanosleep(ns); ns = ns < 256 ? 2 * ns : 256; }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (v[u] == 0) v[u] = ld_acquire_i32(lev1 + kk[u]);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) mx = max(mx, v[u]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) st_release_i32(lev1 + j, mx + 1);   // level(j) = mx, stored + 1
        mymax = max(mymax, mx);
    }
    if (lane == 0) atomicMax(maxlev, mymax);
}
// rows per level, from lev1 (level + 1)
__global__ void k_level_count(int64_t n, const int* lev1, unsigned long long* cnt) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(cnt + (lev1[j] - 1), 1ull);
}
// slot of every row: its level's offset plus a cursor (order inside a level is free)
__global__ void k_level_scatter(int64_t n, const int* lev1, const int64_t* off, unsigned long long* cur,
                                int32_t* sched) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const int l = lev1[j] - 1;
        const int64_t at = off[l] + (int64_t)atomicAdd(cur + l, 1ull);
        sched[at] = (int32_t)j;
    }
}

// lev1 of one direction by the row form, and the deepest level
template <bool FWD>
static lsq_status levels_by_row(const SparseHandle* S, int64_t n, int* lev1, int* maxlev, unsigned* err, cudaStream_t st) {
    int dev = 0, sms = 0, per = 0;
    LSQ_CUDA(cudaGetDevice(&dev));
    LSQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    LSQ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_levels<FWD>, 256, 0));
    if (per < 1) { set_error("level kernel does not fit on an SM"); return LSQ_ERR_CUDA; }
    int64_t nn = n;
    const int64_t* mptr = S->mptr;
    const int32_t* mcol = S->mcol;
    const int64_t* mdiag = S->mdiag;
    unsigned max_polls = dep_wait_polls();
    void* params[] = {&nn, (void*)&mptr, (void*)&mcol, (void*)&mdiag, &lev1, &maxlev, &err, &max_polls};
    LSQ_CUDA(cudaLaunchCooperativeKernel((const void*)k_levels<FWD>, dim3(sms * per), dim3(256), params, 0, st));
    count_launch();
    return LSQ_OK;
}
// One direction's schedule from its levels: sched (n rows, level by level) and loff (L + 1
// offsets into sched).
static lsq_status level_schedule(int64_t n, const int* lev1, int64_t L, int32_t** sched, int64_t** loff,
                                 cudaStream_t st) {
    LSQ_CUDA(pool_alloc(sched, 4 * (size_t)n, st));
    LSQ_CUDA(pool_alloc(loff, 8 * (size_t)(L + 1), st));
    Scratch sc2;
    const int64_t nt = (L + SC_T - 1) / SC_T;   // scan_i64: out[0..L], ceil(L / 512) scratch
    LSQ_CUDA(sc2.alloc(8 * (size_t)(2 * L + nt + 1), st));
    int64_t* lsize = sc2.as<int64_t>();         // rows per level
    unsigned long long* cur = reinterpret_cast<unsigned long long*>(lsize + L);
    int64_t* scan_scratch = lsize + 2 * L;
    LSQ_CUDA(cudaMemsetAsync(lsize, 0, 16 * (size_t)L, st));
    k_level_count<<<grid1(n), 256, 0, st>>>(n, lev1, reinterpret_cast<unsigned long long*>(lsize));
    count_launch();
    lsq_status r = scan_i64(lsize, L, *loff, scan_scratch, st);
    if (r != LSQ_OK) return r;
    k_level_scatter<<<grid1(n), 256, 0, st>>>(n, lev1, *loff, cur, *sched);
    count_launch();
    LSQ_CUDA(cudaGetLastError());
    return LSQ_OK;
}
// Both directions' schedules on the device.  The levels come from the chain of 128-row blocks
// where rows are long against it (a random M with d dependencies per row is about 4 d levels
// deep, and the row form pays for every level), from the row form otherwise.
// 40,000 rows with 380 dependencies each (1583 levels, 313 blocks): 27.7 ms
// by rows, 1.8 ms by blocks (both directions).
static lsq_status device_levels(SparseHandle* S, int64_t n, int64_t nnz_m, cudaStream_t st) {
    Scratch sc;
    LSQ_CUDA(sc.alloc(8 * (size_t)n + 256, st));
    int* lev_f = sc.as<int>();
    int* lev_b = lev_f + n;
    int* mx = lev_b + n;                        // deepest levels, then the error word
    unsigned* err = reinterpret_cast<unsigned*>(mx + 2);
    LSQ_CUDA(cudaMemsetAsync(lev_f, 0, 8 * (size_t)n + 256, st));
    const double dep = (double)(nnz_m - n) / (2.0 * (double)n);
    lsq_status r;
    if (dep * 512.0 > (double)n) {
        r = sb_levels(S, n, lev_f, lev_b, mx, mx + 1, err, st);
        if (r != LSQ_OK) return r;
    } else {
        r = levels_by_row<true>(S, n, lev_f, mx, err, st);
        if (r != LSQ_OK) return r;
        r = levels_by_row<false>(S, n, lev_b, mx + 1, err, st);
        if (r != LSQ_OK) return r;
    }
    int hm[3] = {0, 0, 0};
    LSQ_CUDA(cudaMemcpyAsync(hm, mx, 12, cudaMemcpyDeviceToHost, st));
    LSQ_CUDA(cudaStreamSynchronize(st));
    if (hm[2] != 0) { set_error("level schedule: a dependency wait timed out"); return LSQ_ERR_TIMEOUT; }
    S->nlev_f = (int64_t)hm[0] + 1;
    S->nlev_b = (int64_t)hm[1] + 1;
    r = level_schedule(n, lev_f, S->nlev_f, &S->sched_f, &S->loff_f, st);
    if (r != LSQ_OK) return r;
    return level_schedule(n, lev_b, S->nlev_b, &S->sched_b, &S->loff_b, st);
}

lsq_status build_sparse(const lsq_matrix* A, const int32_t* idx, const double* p, int64_t s,
                        lsq_precond* H, cudaStream_t st) {
    const int64_t m = A->m, n = A->n;
    SparseHandle* S = new SparseHandle();
    H->sp = S;
    // 1. compaction
    Scratch sc1;
    const int64_t ntm = (m + SC_T - 1) / SC_T + 1;
    Carve c1;
    c1.add(8 * (size_t)m); c1.add(8 * (size_t)m); c1.add(8 * (size_t)m); c1.add(8 * (size_t)(m + 1));
    c1.add(8 * (size_t)ntm);
    LSQ_CUDA(sc1.alloc(c1.total(), st));
    int64_t* cnt = (int64_t*)c1.at(sc1.as<char>(), 0);
    double* prob = (double*)c1.at(sc1.as<char>(), 1);
    int64_t* flag = (int64_t*)c1.at(sc1.as<char>(), 2);
    int64_t* pos = (int64_t*)c1.at(sc1.as<char>(), 3);   // m + 1
    int64_t* ts = (int64_t*)c1.at(sc1.as<char>(), 4);
    LSQ_CUDA(cudaMemsetAsync(cnt, 0, 8 * (size_t)m, st));
    k_count_draws<<<grid1(s), 256, 0, st>>>(idx, p, s, cnt, prob);
    k_flag<<<grid1(m), 256, 0, st>>>(cnt, m, flag);
    count_launch(2);
    lsq_status r = scan_i64(flag, m, pos, ts, st);
    if (r != LSQ_OK) return r;
    int64_t nu = 0;
    LSQ_CUDA(cudaMemcpyAsync(&nu, pos + m, 8, cudaMemcpyDeviceToHost, st));
    LSQ_CUDA(cudaStreamSynchronize(st));
    Scratch sc2;
    const int64_t ntu = (nu + SC_T - 1) / SC_T + 1;
    Carve c2;
    c2.add(4 * (size_t)nu); c2.add(8 * (size_t)nu); c2.add(8 * (size_t)nu); c2.add(8 * (size_t)(nu + 1));
    c2.add(8 * (size_t)ntu);
    LSQ_CUDA(sc2.alloc(c2.total(), st));
    int32_t* urow = (int32_t*)c2.at(sc2.as<char>(), 0);
    double* gam = (double*)c2.at(sc2.as<char>(), 1);
    int64_t* ulen = (int64_t*)c2.at(sc2.as<char>(), 2);
    int64_t* sptr = (int64_t*)c2.at(sc2.as<char>(), 3);   // nu + 1
    int64_t* ts2 = (int64_t*)c2.at(sc2.as<char>(), 4);
    k_compact<<<grid1(m), 256, 0, st>>>(cnt, prob, pos, m, s, A->row_ptr, urow, gam, ulen);
    count_launch();
    r = scan_i64(ulen, nu, sptr, ts2, st);
    if (r != LSQ_OK) return r;
    int64_t snnz = 0;
    LSQ_CUDA(cudaMemcpyAsync(&snnz, sptr + nu, 8, cudaMemcpyDeviceToHost, st));
    LSQ_CUDA(cudaStreamSynchronize(st));
    // 2. A_s and its transpose
    Scratch sc3;
    Carve c3;
    c3.add(4 * (size_t)snnz); c3.add(8 * (size_t)snnz); c3.add(8 * (size_t)(n + 1));
    c3.add(4 * (size_t)snnz); c3.add(8 * (size_t)snnz);
    LSQ_CUDA(sc3.alloc(c3.total(), st));
    int32_t* scol = (int32_t*)c3.at(sc3.as<char>(), 0);
    double* sval = (double*)c3.at(sc3.as<char>(), 1);
    int64_t* tptr = (int64_t*)c3.at(sc3.as<char>(), 2);
    int32_t* trow = (int32_t*)c3.at(sc3.as<char>(), 3);
    int64_t* tperm = (int64_t*)c3.at(sc3.as<char>(), 4);
    switch (A->dtype) {
        case LSQ_F64: k_fill_As<LSQ_F64><<<grid1(nu * 32), 256, 0, st>>>(*A, urow, nu, sptr, H->inv_d, scol, sval); break;
        case LSQ_F32: k_fill_As<LSQ_F32><<<grid1(nu * 32), 256, 0, st>>>(*A, urow, nu, sptr, H->inv_d, scol, sval); break;
        case LSQ_BF16: k_fill_As<LSQ_BF16><<<grid1(nu * 32), 256, 0, st>>>(*A, urow, nu, sptr, H->inv_d, scol, sval); break;
        default: k_fill_As<LSQ_F32X2><<<grid1(nu * 32), 256, 0, st>>>(*A, urow, nu, sptr, H->inv_d, scol, sval); break;
    }
    count_launch();
    r = transpose_pattern(sptr, scol, nu, n, snnz, tptr, trow, tperm, st);
    if (r != LSQ_OK) return r;
    // 3. SpGEMM: candidates, counts, row pointers, values
    Scratch sc4;
    int64_t ntn = (n + SC_T - 1) / SC_T + 1;
    LSQ_CUDA(sc4.alloc(8 * (size_t)(n + 16 + ntn) + 4 * (size_t)n, st));
    int64_t* mcnt = sc4.as<int64_t>();
    unsigned long long* nfix = reinterpret_cast<unsigned long long*>(mcnt + n);
    int* mmax = reinterpret_cast<int*>(nfix + 1);   // most candidates and most entries of a row
    int64_t* ts4 = mcnt + n + 16;
    int32_t* cand = reinterpret_cast<int32_t*>(ts4 + ntn);
    LSQ_CUDA(cudaMemsetAsync(nfix, 0, 32, st));
    LSQ_CUDA(pool_alloc(&S->mptr, 8 * (size_t)(n + 1), st));
    int dev = 0, sms = 0;
    LSQ_CUDA(cudaGetDevice(&dev));
    LSQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    k_spg_cand<<<grid1(n * 32), 256, 0, st>>>(n, sptr, tptr, trow, cand, mmax);
    count_launch();
    int hmax[2] = {0, 0};
    LSQ_CUDA(cudaMemcpyAsync(hmax, mmax, 4, cudaMemcpyDeviceToHost, st));
    LSQ_CUDA(cudaStreamSynchronize(st));
    if (hmax[0] > SPG_CAP) {
        set_error("a row of A_s^T A_s has more than 8192 candidate products (unsupported in this build)");
        return LSQ_ERR_UNSUPPORTED;
    }
    SpgArgs ga{};
    ga.n = n; ga.sptr = sptr; ga.scol = scol; ga.sval = sval; ga.gam = gam;
    ga.tptr = tptr; ga.trow = trow; ga.tperm = tperm; ga.cand = cand;
    ga.mcnt = mcnt; ga.maxrow = mmax + 1; ga.n_fixed = nfix;
    r = spgemm_pass<false>(ga, hmax[0], sms, st);
    if (r != LSQ_OK) return r;
    r = scan_i64(mcnt, n, S->mptr, ts4, st);
    if (r != LSQ_OK) return r;
    int64_t mnnz = 0;
    LSQ_CUDA(cudaMemcpyAsync(&mnnz, S->mptr + n, 8, cudaMemcpyDeviceToHost, st));
    LSQ_CUDA(cudaMemcpyAsync(hmax, mmax, 8, cudaMemcpyDeviceToHost, st));
    LSQ_CUDA(cudaStreamSynchronize(st));
    LSQ_CUDA(pool_alloc(&S->mcol, 4 * (size_t)mnnz, st));
    LSQ_CUDA(pool_alloc(&S->mval, 8 * (size_t)mnnz, st));
    if (H->op_dtype == LSQ_F32) LSQ_CUDA(pool_alloc(&S->mval32, 4 * (size_t)mnnz, st));
    LSQ_CUDA(pool_alloc(&S->dinv, 8 * (size_t)n, st));
    LSQ_CUDA(pool_alloc(&S->mdiag, 8 * (size_t)n, st));
    ga.mptr = S->mptr; ga.mcol = S->mcol; ga.mval = S->mval; ga.mval32 = S->mval32;
    ga.dinv = S->dinv; ga.mdiag = S->mdiag; ga.acap = (hmax[1] + 1) & ~1;
    r = spgemm_pass<true>(ga, hmax[0], sms, st);
    if (r != LSQ_OK) return r;
    unsigned long long nf = 0;
    LSQ_CUDA(cudaMemcpyAsync(&nf, nfix, 8, cudaMemcpyDeviceToHost, st));
    LSQ_CUDA(cudaGetLastError());
    LSQ_CUDA(cudaStreamSynchronize(st));
    S->nnz_M = mnnz;
    // 4. level schedules of the forward and backward sweeps (device)
    r = device_levels(S, n, mnnz, st);
    if (r != LSQ_OK) return r;
    if (H->sweeps > 0) {   // t = 0 (the identity) sweeps nothing
        r = sb_build_inverse(S, n, H->op_dtype == LSQ_F32, st);
        if (r != LSQ_OK) return r;
    }
    // 5. transposed pattern of A for the A^T q pass (values are gathered at solve time)
    LSQ_CUDA(pool_alloc(&S->atptr, 8 * (size_t)(n + 1), st));
    LSQ_CUDA(pool_alloc(&S->atrow, 4 * (size_t)A->nnz, st));
    LSQ_CUDA(pool_alloc(&S->atperm, 8 * (size_t)A->nnz, st));
    r = transpose_pattern(A->row_ptr, A->col_idx, m, n, A->nnz, S->atptr, S->atrow, S->atperm, st);
    if (r != LSQ_OK) return r;
    LSQ_CUDA(cudaStreamSynchronize(st));
    S->nnz_A = A->nnz;
    S->m = m;
    H->n_fixed_diag = (int64_t)nf;
    H->nnz_M = mnnz;
    H->levels = S->nlev_f;
    S->n_unique = nu;
    return LSQ_OK;
}

void free_sparse(SparseHandle* S, int device) {
    if (!S) return;
    pool_free(device, {S->mptr, S->mcol, S->mval, S->mval32, S->dinv, S->mdiag, S->sched_f, S->sched_b, S->inv,
                       S->atptr, S->atrow, S->atperm, S->loff_f, S->loff_b});
    delete S;
}

}  // namespace lsq
