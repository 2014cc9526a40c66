// Gauss-Seidel sweeps of Alg. 3 by blocks of B consecutive rows, for deep level schedules.
//
// A forward sweep solves (D + L) x = s for s = r - U e_old in the natural row order.  With the
// rows in blocks, block k needs x of the blocks before it; inside the block the triangular
// system is solved by one product with the block's inverse, computed once per handle:
//     x_k = (D + L)_kk^{-1} (s_k - sum_{i < k} L_ki x_i).
// The chain of a sweep is then n / B blocks instead of the level schedule's depth.  A CTA owns
// blocks k, k + G, ...; it follows the blocks before its own one after the other: it waits for
// their B values (the values are their own completion flags, as in the row forms: a slot holds
// SB_EMPTY until it is written), puts them in shared memory, and every thread adds up the
// entries of its row that fall in them (rows are sorted, so a thread's cursor only moves on).
// Behind the last of them only the reduction of ES partial sums and the B x B product stand
// between two blocks.  A block that starts late finds the first blocks finished and takes four
// at a time until it has caught up.
//
// Bound: the chain's latency: the values' way to another SM, the last entries, the reduction of
// ES sums and the product.  The inverse sits in registers (each thread holds the part of its row
// it multiplies), loaded while the CTA waits.
// Measured per sweep: 40,000 rows of 380 dependencies in 1583 levels, one column, double-float:
// 0.54 ms (1.7 us per block of 128 rows), against 1.75 ms forward and 3.5 ms backward by rows;
// 10,000 rows of 350 dependencies in 1227 levels, 16 columns: 0.42 ms (2.7 us per block of 64),
// against 5.3 and 6.1 ms.
// Columns are independent chains, so a block of right-hand sides is split over CTAs by KC
// columns.
//
// Waits are bounded as everywhere: one that gives up sets the error word, which ends the others.
// Every CTA is resident (cooperative launch) and takes its blocks in increasing order, so every
// wait ends.
#include "sweep_blocked.cuh"
#include "dfloat.cuh"

#include <algorithm>
#include <mutex>
#include <unordered_map>

namespace lsq {

constexpr unsigned long long SB_EMPTY = 0xFFF7DEADBEEFCAFEull;   // the row forms' empty marker
constexpr int SB_T = 512;
constexpr int SB_SPAN = 4;          // blocks taken at once while catching up
constexpr unsigned SB_FAR_NS = 100; // between the polls of a CTA that is far behind its block

__device__ __forceinline__ unsigned long long sb_ldv(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.volatile.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void sb_stv(unsigned long long* p, unsigned long long v) {
    asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// one 4- or 8-byte element global -> shared, asynchronously
template <typename T>
__device__ __forceinline__ void cp_async_elem(T* dst, const T* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (sizeof(T) == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// Arithmetic of a sweep: double-float pairs for FP32 M, or FP64 sums for either type of M.
struct SbPair {
    typedef f2 V;
    static __device__ __forceinline__ V zero() { return f2{0.f, 0.f}; }
    static __device__ __forceinline__ V from_bits(unsigned long long u) {
        return f2{__uint_as_float((unsigned)u), __uint_as_float((unsigned)(u >> 32))};
    }
    static __device__ __forceinline__ unsigned long long to_bits(V v) {
        return (unsigned long long)__float_as_uint(v.hi) | ((unsigned long long)__float_as_uint(v.lo) << 32);
    }
    static __device__ __forceinline__ V from_double(double x) { return df_from_double(x); }
    static __device__ __forceinline__ double to_double(V v) { return df_to_double(v); }
    // acc += m x, cascaded (the errors gather in the low word)
    static __device__ __forceinline__ void mad(V& acc, float m, V x) {
        float p, pe, s, e;
        two_prod(m, x.hi, p, pe);
        pe = fmaf(m, x.lo, pe);
        two_sum(acc.hi, p, s, e);
        acc.hi = s;
        acc.lo += e + pe;
    }
    static __device__ __forceinline__ void madv(V& acc, V m, V x) { df_fma_cascade(acc, m, x); }
    static __device__ __forceinline__ void norm(V& v) { v = df_norm(v); }
    static __device__ __forceinline__ void add(V& a, V b) { df_add(a, b); }
    static __device__ __forceinline__ V xorv(V v, int o) { return df_shfl_xor(v, o); }
    static __device__ __forceinline__ V neg(V v) { return f2{-v.hi, -v.lo}; }
};
struct SbDouble {
    typedef double V;
    static __device__ __forceinline__ V zero() { return 0.0; }
    static __device__ __forceinline__ V from_bits(unsigned long long u) { return __longlong_as_double((long long)u); }
    static __device__ __forceinline__ unsigned long long to_bits(V v) { return (unsigned long long)__double_as_longlong(v); }
    static __device__ __forceinline__ V from_double(double x) { return x; }
    static __device__ __forceinline__ double to_double(V v) { return v; }
    static __device__ __forceinline__ void mad(V& acc, double m, V x) { acc = fma(m, x, acc); }
    static __device__ __forceinline__ void madv(V& acc, V m, V x) { acc = fma(m, x, acc); }
    static __device__ __forceinline__ void norm(V&) {}
    static __device__ __forceinline__ void add(V& a, V b) { a += b; }
    static __device__ __forceinline__ V xorv(V v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
    static __device__ __forceinline__ V neg(V v) { return -v; }
};

// MT: type of M's values; AR: arithmetic; B rows per block, KC columns per CTA.  Thread (row, h, c) of the 512 owns
// entries h, h + ES, ... of its row for column c.
template <typename MT, typename AR, bool FWD, int B, int KC>
__global__ void __launch_bounds__(SB_T, 1) k_sweep_blocked(SbArgs a) {
    typedef typename AR::V V;
    constexpr int ES = SB_T / (B * KC);
    constexpr int PER = B / ES;          // inverse entries per thread
    static_assert(ES >= 1 && ES * KC <= 32 && SB_ROWS % B == 0, "thread layout");
    __shared__ V s_x[2][SB_SPAN * B * KC];
    __shared__ V s_s[B * KC];
    constexpr int AHEAD = sizeof(MT) == 4 ? 6 : 4;       // entries under way per thread
    __shared__ int s_qc[AHEAD][SB_T];
    __shared__ MT s_qv[AHEAD][SB_T];
    __shared__ double s_red[SB_T / 32];
    __shared__ int s_stop;
    if (*a.done) return;
    const int tid = threadIdx.x, lane = tid & 31;
    if (a.S) {   // the convergence check of the one-column solve, the same decision in every CTA
        double t = 0.0;
        for (int i = tid; i < a.nparts; i += SB_T) t += a.part[i];
        t = warp_sum(t);
        if (lane == 0) s_red[tid >> 5] = t;
        __syncthreads();
        if (tid == 0) {
            double gg = 0.0;
            for (int w = 0; w < SB_T / 32; ++w) gg += s_red[w];
            const double gn = sqrt(gg);
            s_stop = (gn <= a.tol * a.S->hn || gn <= a.inner_tol * a.S->gstart || a.S->iters >= a.maxit) ? 1 : 0;
            if (blockIdx.x == 0) a.S->rec = gn / a.S->hn;
        }
        __syncthreads();
        if (s_stop) {
            if (blockIdx.x == 0 && tid == 0) a.S->done = 1;
            return;
        }
    }
    const MT* __restrict__ mv = reinterpret_cast<const MT*>(a.mval);
    const int32_t* __restrict__ mc = a.mcol;
    unsigned long long* xnew = reinterpret_cast<unsigned long long*>(a.e_new);
    const unsigned long long* xold = reinterpret_cast<const unsigned long long*>(a.e_old);
    // a warp takes RW consecutive rows; the row groups are dealt so that the triangles of the four
    // schedulers (warps s, s + 4, s + 8, s + 12) are the same size
    constexpr int RW = 32 / (KC * ES);
    const int wg = (tid >> 7) & 3, wsch = (tid >> 5) & 3;
    const int wrow0 = RW * (wg * 4 + ((wg & 1) ? 3 - wsch : wsch)), wrow1 = wrow0 + RW - 1;
    const int c = tid % KC, h = (tid / KC) % ES, row = wrow0 + lane / (KC * ES);
    const int nblk = (int)((a.n + B - 1) / B);
    const int ngrp = (a.K + KC - 1) / KC;
    const int64_t ntask = (int64_t)nblk * ngrp;
    for (int64_t task = blockIdx.x; task < ntask; task += gridDim.x) {
        const int kk = (int)(task / ngrp), cg = (int)(task % ngrp);
        const int kb = FWD ? kk : nblk - 1 - kk;          // this block
        const int64_t j = (int64_t)kb * B + row;
        const int col = cg * KC + c;
        const bool live = j < a.n && col < a.K;
        // the part of the inverse this thread multiplies: entries h, h + ES, ... of its row
        // (backward: M is symmetric, so the upper block's inverse is the transpose)
        V inv[PER];
        {
            const int sub = (kb * B) % SB_ROWS;           // place inside the stored block
            const int64_t at = (int64_t)((int64_t)kb * B / SB_ROWS) * SB_ROWS * SB_ROWS;
            const int ri = sub + row;
#pragma unroll
            for (int t = 0; t < PER; ++t) {
                const int ci = sub + h + ES * t;
                const int64_t e = at + (FWD ? (int64_t)ri * SB_ROWS + ci : (int64_t)ci * SB_ROWS + ri);
                if constexpr (std::is_same<AR, SbPair>::value) {
                    if (!a.inv64) inv[t] = reinterpret_cast<const f2*>(a.inv)[e];
                    else inv[t] = df_from_double(reinterpret_cast<const double*>(a.inv)[e]);
                } else {
                    inv[t] = reinterpret_cast<const double*>(a.inv)[e];
                }
            }
        }
        // base term, the other side's terms (previous sweep: complete), and the cursor
        V acc = AR::zero(), base = AR::zero();
        int64_t e = 0, e_end = 0;
        if (live) {
            const int64_t p0 = a.mptr[j], pd = a.mdiag[j], p1 = a.mptr[j + 1];
            if (a.identity) {      // r - L e_old = D e_old after one forward sweep from zero
                if (h == 0) AR::madv(base, AR::from_double(a.mval64[pd]), AR::from_bits(xold[j * a.K + col]));
            } else {
                if (h == 0) base = AR::from_double(a.r[j * a.K + col]);
                if (a.e_old) {
                    const int64_t o0 = FWD ? pd + 1 : p0, o1 = FWD ? p1 : pd;
                    for (int64_t q = o0 + h; q < o1; q += ES)
                        AR::mad(acc, mv[q], AR::from_bits(xold[(int64_t)mc[q] * a.K + col]));
                }
            }
            if (FWD) { e = p0 + h; e_end = pd; }
            else { e = p1 - 1 - h; e_end = pd; }
        }
        // The cursor: this thread's entries of M, AHEAD of them under way to its own slots of
        // shared memory.  M streams from L2 or HBM, and an entry waited for inside the walk stands in
        // the chain; a queue in registers waits as well, because moving a register up needs the load
        // that fills it.  A column past every block ends the walk.
        constexpr int PAST = FWD ? 0x7fffffff : -1;
        auto fetch = [&](int at) {
            const bool in = FWD ? e < e_end : e > e_end;
            if (in) {
                cp_async_elem(&s_qc[at][tid], mc + e);
                cp_async_elem(&s_qv[at][tid], mv + e);
                e += FWD ? ES : -ES;
            } else {
                s_qc[at][tid] = PAST;
            }
        };
        asm volatile("cp.async.wait_group 0;" ::: "memory");   // the last block's left-over entries
        if (!live) e = e_end = 0;
#pragma unroll
        for (int q = 0; q < AHEAD; ++q) {
            fetch(q);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        int head = 0;
        asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory");
        int cc = s_qc[0][tid];
        MT cv = s_qv[0][tid];
        // slot of this thread's value in block i of the chain (i-th block done)
        const int lrow = tid / KC;
        auto slot = [&](int i) -> const unsigned long long* {
            const int64_t jj = (int64_t)(FWD ? i : nblk - 1 - i) * B + lrow;
            return (tid < B * KC && jj < a.n && col < a.K) ? xnew + jj * a.K + cg * KC + tid % KC : nullptr;
        };
        int i = 0, buf = 0;
        while (i < kk) {
            // Far behind its own block the CTA takes four blocks at a time, and one thread waits
            // for the last of them, now and then; only the CTAs of the next few blocks watch every
            // value.  (All CTAs polling all values kept the chain's own stores waiting.)
            const int span = kk - i > SB_SPAN ? SB_SPAN : 1;
            if (span > 1) {
                if (tid == 0) {
                    const int64_t j3 = (int64_t)(FWD ? i + span - 1 : nblk - i - span) * B;
                    const unsigned long long* p = xnew + j3 * a.K + cg * KC;
                    unsigned polls = 0;
                    while (sb_ldv(p) == SB_EMPTY) {
                        ++polls;
                        if (polls > a.max_polls || ((polls & 63u) == 0 && *(volatile unsigned*)a.err != 0u)) {
                            atomicOr(a.err, DEV_ERR_TIMEOUT);
                            break;
                        }
                        __nanosleep(SB_FAR_NS);
                    }
                }
                __syncthreads();
            }
            if (tid < ((B * KC + 31) & ~31)) {
                unsigned long long u[SB_SPAN];
#pragma unroll
                for (int q = 0; q < SB_SPAN; ++q) {
                    const unsigned long long* p = q < span ? slot(i + q) : nullptr;
                    u[q] = p ? sb_ldv(p) : 0ull;
                }
                unsigned polls = 0;
                while (true) {
                    bool missing = false;
#pragma unroll
                    for (int q = 0; q < SB_SPAN; ++q) missing = missing || u[q] == SB_EMPTY;
                    if (!__any_sync(0xffffffffu, missing)) break;
                    ++polls;
                    const bool give_up = polls > a.max_polls ||
                                         ((polls & 255u) == 0 && *(volatile unsigned*)a.err != 0u);
                    if (__any_sync(0xffffffffu, give_up)) {
                        if (lane == 0) atomicOr(a.err, DEV_ERR_TIMEOUT);
#pragma unroll
                        for (int q = 0; q < SB_SPAN; ++q)
                            if (u[q] == SB_EMPTY) u[q] = 0ull;
                        break;
                    }
                    if (polls > 64) __nanosleep(polls > 4096 ? 128 : 20);
#pragma unroll
                    for (int q = 0; q < SB_SPAN; ++q)
                        if (u[q] == SB_EMPTY) u[q] = sb_ldv(slot(i + q));
                }
#pragma unroll
                for (int q = 0; q < SB_SPAN; ++q)
                    if (q < span && tid < B * KC) s_x[buf][q * B * KC + tid] = AR::from_bits(u[q]);
            }
            __syncthreads();
            // this thread's entries inside the blocks just loaded
            const int64_t first = (int64_t)(FWD ? i : nblk - i - span) * B;   // lowest row of the span
            const int lim = FWD ? (int)min(first + (int64_t)span * B, (int64_t)0x7fffffff) : (int)first;
            while (true) {
                // the warp goes round as one until no lane has an entry left in the span
                const bool on = FWD ? cc < lim : cc >= lim;
                if (!__any_sync(0xffffffffu, on)) break;
                if (on) {
                    const int d = cc - (int)first;
                    // forward: block q of the span starts at q B; backward: the span runs downwards
                    const int at = FWD ? d : (span - 1 - d / B) * B + (d & (B - 1));
                    AR::mad(acc, cv, s_x[buf][at * KC + c]);
                    fetch(head);
                    head = head + 1 == AHEAD ? 0 : head + 1;
                }
                asm volatile("cp.async.commit_group;\n\tcp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory");
                if (on) {
                    cc = s_qc[head][tid];
                    cv = s_qv[head][tid];
                }
            }
            i += span;
            buf ^= 1;
        }
        __syncwarp();
        // s_row = base - sum over the row's ES threads
        AR::norm(acc);
        V s = AR::neg(acc);
        if (h == 0) { AR::norm(base); AR::add(s, base); }
#pragma unroll
        for (int o = KC; o < KC * ES; o <<= 1) AR::add(s, AR::xorv(s, o));
        if (h == 0) s_s[row * KC + c] = s;
        __syncthreads();
        // x_row = sum_k inv(row, k) s_k over the triangle, CH entries at a time; the warp skips the
        // chunks that are zero for all of its rows.  (A test per entry left every entry's shared
        // load and multiply-add waiting for the one before: 2900 cycles of a 5000-cycle step.)
        constexpr int CH = std::is_same<AR, SbPair>::value ? 8 : (PER >= 16 ? 4 : 2);
        V x = AR::zero();
#pragma unroll
        for (int t0 = 0; t0 < PER; t0 += CH) {
            const bool need = FWD ? ES * t0 <= wrow1 : ES * (t0 + CH) - 1 >= wrow0;
            if (need) {
                V sv[CH];
#pragma unroll
                for (int t = 0; t < CH; ++t) sv[t] = s_s[(h + ES * (t0 + t)) * KC + c];
#pragma unroll
                for (int t = 0; t < CH; ++t) AR::madv(x, inv[t0 + t], sv[t]);
            }
        }
        AR::norm(x);
#pragma unroll
        for (int o = KC; o < KC * ES; o <<= 1) AR::add(x, AR::xorv(x, o));
        if (h == 0 && live) {
            sb_stv(xnew + j * a.K + col, AR::to_bits(x));
            if (a.out64) a.out64[j * a.K + col] = AR::to_double(x);
        }
        __syncthreads();   // s_s and s_x are reused by the next block
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");   // the last block's left-over entries
}

// ---------------------------------------------------------------------------------------
// Inverses of the 128-row lower diagonal blocks D + L of M: the block in shared memory (M's
// entries, the identity beyond n), inverted in place from the last column to the first
// (column j of the inverse is -X_sub l_j / l_jj with X_sub the inverse of the rows below),
// four threads per row.  FP64 throughout, from the FP32-rounded off-diagonal entries and the FP64
// diagonal for FP32 M.  Stored as doubles, or as float pairs where every sweep that uses them runs in
// double-float.
// Bound: FP64 instructions (350 k FMAs per block and as many lanes again in the row reductions; the
// reciprocals of the diagonal are formed once: a division per thread and column took most of the
// time).  313 blocks: 0.71 ms, against
// 1.56 ms.
// ---------------------------------------------------------------------------------------
constexpr int SI_LD = SB_ROWS + 1;
constexpr int SI_T = 512;
constexpr size_t SI_SMEM = (size_t)SB_ROWS * SI_LD * 8;
template <typename MT>
__global__ void __launch_bounds__(SI_T, 1) k_block_inverse(int64_t n, const int64_t* mptr, const int32_t* mcol,
                                                           const MT* mval, const double* mval64,
                                                           const int64_t* mdiag, void* inv, int inv64) {
    extern __shared__ __align__(16) double s_a[];   // SB_ROWS x SI_LD, row-major
    __shared__ double s_l[SB_ROWS], s_rd[SB_ROWS];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nblk = (int)((n + SB_ROWS - 1) / SB_ROWS);
    for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
        const int64_t j0 = (int64_t)b * SB_ROWS;
        for (int t = tid; t < SB_ROWS * SI_LD; t += SI_T) s_a[t] = 0.0;
        __syncthreads();
        for (int r = wid; r < SB_ROWS; r += SI_T / 32) {
            const int64_t j = j0 + r;
            if (j >= n) {
                if (lane == 0) s_a[r * SI_LD + r] = 1.0;
                continue;
            }
            const int64_t ed = mdiag[j], e0 = mptr[j];
            if (lane == 0) s_a[r * SI_LD + r] = mval64[ed];
            for (int64_t e = ed - 1 - lane; e >= e0; e -= 32) {   // sorted: leave below the block
                const int32_t k = mcol[e];
                if (k < j0) break;
                s_a[r * SI_LD + (int)(k - j0)] = (double)mval[e];
            }
        }
        __syncthreads();
        if (tid < SB_ROWS) s_rd[tid] = 1.0 / s_a[tid * SI_LD + tid];
        const int row = tid >> 2, h = tid & 3;
        for (int j = SB_ROWS - 1; j >= 0; --j) {
            if (tid < SB_ROWS) s_l[tid] = s_a[tid * SI_LD + j];
            __syncthreads();
            // warps whose rows all lie at or above j have nothing to do (eight rows a warp)
            if ((row | 7) > j) {
                double t = 0.0;
                if (row > j)
                    for (int k = j + 1 + h; k <= row; k += 4) t = fma(s_a[row * SI_LD + k], s_l[k], t);
                t += __shfl_xor_sync(0xffffffffu, t, 1);
                t += __shfl_xor_sync(0xffffffffu, t, 2);
                if (h == 0 && row > j) s_a[row * SI_LD + j] = -t * s_rd[j];
            }
            if (tid == 0) s_a[j * SI_LD + j] = s_rd[j];
            __syncthreads();
        }
        for (int t = tid; t < SB_ROWS * SB_ROWS; t += SI_T) {
            const double v = s_a[(t / SB_ROWS) * SI_LD + t % SB_ROWS];
            const int64_t at = (int64_t)b * SB_ROWS * SB_ROWS + t;
            if (inv64) reinterpret_cast<double*>(inv)[at] = v;
            else reinterpret_cast<f2*>(inv)[at] = df_from_double(v);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------
// Level of every row by the same chain of blocks: lev1(j) = 1 + max lev1 over the row's
// dependencies (1 without any); 0 = not yet known.  Dependencies in earlier blocks are
// followed as in the sweep; inside the block the rows are relaxed until nothing changes
// (as many rounds as the block's own depth).  Even CTAs take the forward direction, odd ones the
// backward one.
// ---------------------------------------------------------------------------------------
constexpr int SL_T = 256, SL_AHEAD = 8;
template <bool FWD>
__device__ __forceinline__ void levels_blocked(int64_t n, const int64_t* mptr, const int32_t* mcol,
                                               const int64_t* mdiag, int* lev1, int* maxlev, unsigned* err,
                                               unsigned max_polls, int first_blk, int stride) {
    constexpr int B = SB_ROWS, ES = SL_T / B;
    __shared__ int s_x[2][SB_SPAN * B];
    __shared__ int s_lev[B];
    __shared__ unsigned s_bits[B][B / 32];
    __shared__ int s_qc[SL_AHEAD][SL_T];
    const int tid = threadIdx.x, lane = tid & 31;
    const int row = tid / ES, h = tid % ES;
    const int nblk = (int)((n + B - 1) / B);
    int mymax = 0;
    for (int kk = first_blk; kk < nblk; kk += stride) {
        const int kb = FWD ? kk : nblk - 1 - kk;
        const int64_t j = (int64_t)kb * B + row;
        const int64_t j0 = (int64_t)kb * B;
        int64_t e = 0, e_end = 0;
        if (j < n) {
            e_end = mdiag[j];
            e = FWD ? mptr[j] + h : mptr[j + 1] - 1 - h;
        }
        constexpr int PAST = FWD ? 0x7fffffff : -1;
        if (j >= n) e = e_end = 0;
        auto fetch = [&](int at) {
            const bool in = FWD ? e < e_end : e > e_end;
            if (in) { cp_async_elem(&s_qc[at][tid], mcol + e); e += FWD ? ES : -ES; }
            else s_qc[at][tid] = PAST;
        };
        int head = 0;
        // moves the lanes with `on` to their next entry (the whole warp calls this together)
        auto advance = [&](bool on, int& c0) {
            if (on) {
                fetch(head);
                head = head + 1 == SL_AHEAD ? 0 : head + 1;
            }
            asm volatile("cp.async.commit_group;\n\tcp.async.wait_group %0;" ::"n"(SL_AHEAD - 1) : "memory");
            if (on) c0 = s_qc[head][tid];
        };
        for (int t = tid; t < B * (B / 32); t += SL_T) s_bits[t / (B / 32)][t % (B / 32)] = 0u;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
        for (int q = 0; q < SL_AHEAD; ++q) {
            fetch(q);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        asm volatile("cp.async.wait_group %0;" ::"n"(SL_AHEAD - 1) : "memory");
        int c0 = s_qc[0][tid], mx = 0;
        int buf = 0;
        for (int i = 0; i < kk;) {
            // as in the sweep: far behind, one thread waits for every fourth block
            const int span = kk - i > SB_SPAN ? SB_SPAN : 1;
            if (span > 1) {
                if (tid == 0) {
                    const int* p = lev1 + (int64_t)(FWD ? i + span - 1 : nblk - i - span) * B;
                    unsigned polls = 0;
                    while (*(volatile const int*)p == 0) {
                        ++polls;
                        if (polls > max_polls || ((polls & 63u) == 0 && *(volatile unsigned*)err != 0u)) {
                            atomicOr(err, DEV_ERR_TIMEOUT);
                            break;
                        }
                        __nanosleep(SB_FAR_NS);
                    }
                }
                __syncthreads();
            }
            const int64_t f = (int64_t)(FWD ? i : nblk - i - span) * B;   // lowest row of the span
            if (tid < B) {
                int v[SB_SPAN];
#pragma unroll
                for (int q = 0; q < SB_SPAN; ++q) {
                    const int64_t r = f + q * B + tid;
                    v[q] = q < span && r < n ? *(volatile int*)(lev1 + r) : 1;
                }
                unsigned polls = 0;
                while (true) {
                    bool missing = false;
#pragma unroll
                    for (int q = 0; q < SB_SPAN; ++q) missing = missing || v[q] == 0;
                    if (!__any_sync(0xffffffffu, missing)) break;
                    ++polls;
                    const bool give_up = polls > max_polls || ((polls & 255u) == 0 && *(volatile unsigned*)err != 0u);
                    if (__any_sync(0xffffffffu, give_up)) {
                        if (lane == 0) atomicOr(err, DEV_ERR_TIMEOUT);
#pragma unroll
                        for (int q = 0; q < SB_SPAN; ++q) v[q] = max(v[q], 1);
                        break;
                    }
                    if (polls > 64) __nanosleep(polls > 4096 ? 128 : 20);
#pragma unroll
                    for (int q = 0; q < SB_SPAN; ++q)
                        if (v[q] == 0) v[q] = *(volatile int*)(lev1 + f + q * B + tid);
                }
#pragma unroll
                for (int q = 0; q < SB_SPAN; ++q)
                    if (q < span) s_x[buf][q * B + tid] = v[q];
            }
            __syncthreads();
            const int64_t lim = FWD ? f + (int64_t)span * B : f;
            while (true) {
                const bool on = FWD ? c0 < lim : (c0 >= lim && c0 >= 0);
                if (!__any_sync(0xffffffffu, on)) break;
                if (on) mx = max(mx, s_x[buf][c0 - (int)f]);
                advance(on, c0);
            }
            i += span;
            buf ^= 1;
        }
        __syncwarp();
#pragma unroll
        for (int o = 1; o < ES; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        __syncthreads();   // s_bits cleared
        while (__any_sync(0xffffffffu, c0 != PAST)) {   // what is left of the row lies inside the block
            const bool on = c0 != PAST;
            const int d = c0 - (int)j0;
            if (on) atomicOr(&s_bits[row][d >> 5], 1u << (d & 31));
            advance(on, c0);
        }
        if (h == 0) s_lev[row] = mx + 1;
        __syncthreads();
        unsigned w[B / 32];
        int lv = 0;
        if (tid < B) {
            lv = s_lev[tid];
#pragma unroll
            for (int q = 0; q < B / 32; ++q) w[q] = s_bits[tid][q];
        }
        for (int round = 0; round < B; ++round) {
            int nv = lv;
            if (tid < B) {
#pragma unroll
                for (int q = 0; q < B / 32; ++q) {
                    unsigned m = w[q];
                    while (m) {
                        nv = max(nv, *(volatile int*)&s_lev[q * 32 + __ffs(m) - 1] + 1);
                        m &= m - 1;
                    }
                }
            }
            const bool changed = nv != lv;
            if (changed) { lv = nv; *(volatile int*)&s_lev[tid] = nv; }
            if (!__syncthreads_or(changed)) break;
        }
        if (tid < B && j0 + tid < n) {
            *(volatile int*)(lev1 + j0 + tid) = lv;
            mymax = max(mymax, lv - 1);
        }
        __syncthreads();
    }
    if (mymax > 0) atomicMax(maxlev, mymax);
}
__global__ void __launch_bounds__(SL_T) k_levels_blocked(int64_t n, const int64_t* mptr, const int32_t* mcol,
                                                         const int64_t* mdiag, int* lev1_f, int* lev1_b,
                                                         int* max_f, int* max_b, unsigned* err,
                                                         unsigned max_polls) {
    const int half = gridDim.x >> 1, at = blockIdx.x >> 1;
    if (blockIdx.x & 1) levels_blocked<false>(n, mptr, mcol, mdiag, lev1_b, max_b, err, max_polls, at, half);
    else levels_blocked<true>(n, mptr, mcol, mdiag, lev1_f, max_f, err, max_polls, at, half);
}

// ---------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------
// Resident CTAs of a kernel on the current device (looked up once per kernel and device).
static lsq_status resident_ctas(const void* kern, int threads, size_t smem, int* out) {
    static std::mutex mu;
    static std::unordered_map<const void*, int> known[64];
    int dev = 0;
    LSQ_CUDA(cudaGetDevice(&dev));
    if (dev < 64) {
        std::lock_guard<std::mutex> lk(mu);
        auto it = known[dev].find(kern);
        if (it != known[dev].end()) { *out = it->second; return LSQ_OK; }
    }
    int sms = 0, per = 0;
    LSQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    LSQ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem));
    if (per < 1) { set_error("blocked sweep kernel does not fit on an SM"); return LSQ_ERR_CUDA; }
    *out = sms * per;
    if (dev < 64) {
        std::lock_guard<std::mutex> lk(mu);
        known[dev][kern] = *out;
    }
    return LSQ_OK;
}

// Rows per block and columns per CTA.  Double-float: 128 rows for one column, 64 rows and up to 4
// columns for a block of right-hand sides (the same number of inverse entries per thread).  FP64:
// 64 rows, because the product of a block costs B^2 / 2 FMAs per column at two a clock.
template <typename MT, typename AR, bool FWD>
static const void* sb_kernel(int K, int* B, int* KC) {
    constexpr bool pair = std::is_same<AR, SbPair>::value;
    // one column of FP32 M is always summed in double-float
    if constexpr (pair || sizeof(MT) == 8) {
        if (K == 1) {
            *KC = 1;
            *B = pair ? 128 : 64;
            if constexpr (pair) return (const void*)k_sweep_blocked<MT, AR, FWD, 128, 1>;
            else return (const void*)k_sweep_blocked<MT, AR, FWD, 64, 1>;
        }
    }
    *B = 64;
    if (K <= 2) { *KC = 2; return (const void*)k_sweep_blocked<MT, AR, FWD, 64, 2>; }
    *KC = 4;
    return (const void*)k_sweep_blocked<MT, AR, FWD, 64, 4>;
}

lsq_status sb_launch(const SbArgs& a, bool fwd, bool m32, bool pairs, cudaStream_t st) {
    int B = 0, KC = 0;
    const void* kern;
    if (pairs) kern = fwd ? sb_kernel<float, SbPair, true>(a.K, &B, &KC) : sb_kernel<float, SbPair, false>(a.K, &B, &KC);
    else if (m32) kern = fwd ? sb_kernel<float, SbDouble, true>(a.K, &B, &KC) : sb_kernel<float, SbDouble, false>(a.K, &B, &KC);
    else kern = fwd ? sb_kernel<double, SbDouble, true>(a.K, &B, &KC) : sb_kernel<double, SbDouble, false>(a.K, &B, &KC);
    int res = 0;
    lsq_status r = resident_ctas(kern, SB_T, 0, &res);
    if (r != LSQ_OK) return r;
    const int64_t tasks = (a.n + B - 1) / B * ((a.K + KC - 1) / KC);
    SbArgs av = a;
    void* params[] = {&av};
    LSQ_CUDA(cudaLaunchCooperativeKernel(kern, dim3((unsigned)std::min<int64_t>(tasks, res)), dim3(SB_T), params, 0, st));
    count_launch();
    return LSQ_OK;
}

// The rule: a sweep by blocks takes nblk steps of t_blk, or, with many blocks, the time in which
// the resident CTAs walk all blocks before their own (0.75 us for every four); a sweep by rows takes
// nlev levels of t_row.  Times in us, measured on layers of 40 to 128 nodes with 2 to 110
// dependencies each, 10,000 to 1,000,000 rows:
//   t_blk = base + slope * (entries of a thread in the block before its own),
//   t_row  one column: 1.9 (FP64) or 1.3 (FP32 M) on the grid, 1.2 + 0.22 w or 1.1 + 0.125 w in one CTA,
//          where levels of w rows hold less than 2048 entries; K columns: about 3.5 + 0.14 K with a CTA
//          per row, 2.4 + 0.5 K and, from 4 on, more with the row's length, with a lane per entry.
// At 1,000,000 rows in 10,000 layers of 100, short rows, the walk is the longer of the two (145 ms a sweep
// in FP64, 235 ms in one CTA); at 102,400 rows of 60 dependencies in 1600 layers rows are the
// better form (3.5 ms, blocks 6.5 ms); at 40,000 rows of 380 random dependencies (1583 levels) blocks
// are (0.54 ms, rows 1.75 and 3.5 ms).
bool sb_pays(const SparseHandle* S, int64_t n, int K, bool m32) {
    const double levels = (double)std::min(S->nlev_f, S->nlev_b), dep = (double)(S->nnz_M - n) / (2.0 * (double)n);
    const int mode = block_sweep_mode(S->nnz_M, n);
    if (K > 1 && mode == 0) return false;
    const bool pair = m32 && (K == 1 || mode == 2);
    const int B = K == 1 && pair ? 128 : 64, KC = K == 1 ? 1 : (K == 2 ? 2 : 4), at = KC == 1 ? 0 : (KC == 2 ? 1 : 2);
    static const double base[2][3] = {{2.95, 3.6, 5.4}, {1.75, 2.2, 2.5}};
    static const double slope[2][3] = {{0.145, 0.18, 0.26}, {0.18, 0.13, 0.23}};
    const double nblk = (double)((n + B - 1) / B), groups = (double)((K + KC - 1) / KC);
    const double entries = (B == 128 ? S->near128 : S->near64) * (double)(B * KC) / (double)SB_T;
    const double t_blk = std::max(base[pair][at] + slope[pair][at] * entries, 0.75 * nblk * groups / (4.0 * 2.0 * 152.0));
    double t_row;
    if (K == 1) {
        const double w = (double)n / levels;
        if (dep * w < 2048.0) t_row = m32 ? 1.1 + 0.125 * w : 1.2 + 0.22 * w;
        else t_row = m32 ? 1.3 : 1.9;
    } else if (mode == 2) {
        t_row = 3.5 + 0.14 * K;
    } else {
        t_row = K <= 4 ? 2.4 + 0.5 * K : 4.4 + (K - 4) * (0.25 + 0.0095 * dep);
    }
    return nblk * t_blk <= levels * t_row;
}

// sums over the rows of their entries in the 64-row (sum[0]) and 128-row (sum[1]) block before their own
__global__ void k_near_entries(int64_t n, const int64_t* mptr, const int32_t* mcol, const int64_t* mdiag,
                               unsigned long long* sum) {
    int c[2] = {0, 0};
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p0 = mptr[j], pd = mdiag[j];
        auto first_at = [&](int64_t col) {   // rows are sorted
            int64_t lo = p0, hi = pd;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (mcol[mid] < col) lo = mid + 1;
                else hi = mid;
            }
            return lo;
        };
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int64_t B = 64 << q, b0 = j / B * B;
            c[q] += (int)(first_at(b0) - first_at(b0 - B));
        }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int t = warp_sum(c[q]);
        if ((threadIdx.x & 31) == 0 && t) atomicAdd(&sum[q], (unsigned long long)t);
    }
}

lsq_status sb_build_inverse(SparseHandle* S, int64_t n, bool m32, cudaStream_t st) {
    auto any = [&] {
        return sb_pays(S, n, 1, m32) || sb_pays(S, n, 2, m32) || sb_pays(S, n, 4, m32) || sb_pays(S, n, 16, m32) ||
               sb_pays(S, n, 32, m32);
    };
    if (!any()) return LSQ_OK;   // not even without entries in the block before
    {
        Scratch sc;
        LSQ_CUDA(sc.alloc(16, st));
        LSQ_CUDA(cudaMemsetAsync(sc.ptr, 0, 16, st));
        k_near_entries<<<(unsigned)std::min<int64_t>((n + 255) / 256, 152 * 8), 256, 0, st>>>(
            n, S->mptr, S->mcol, S->mdiag, sc.as<unsigned long long>());
        count_launch();
        unsigned long long sum[2] = {0, 0};
        LSQ_CUDA(cudaMemcpyAsync(sum, sc.ptr, 16, cudaMemcpyDeviceToHost, st));
        LSQ_CUDA(cudaStreamSynchronize(st));
        S->near64 = (double)sum[0] / (double)n;
        S->near128 = (double)sum[1] / (double)n;
    }
    if (!any()) return LSQ_OK;
    const int64_t nblk = (n + SB_ROWS - 1) / SB_ROWS;
    if (pool_alloc(&S->inv, 8 * (size_t)nblk * SB_ROWS * SB_ROWS, st) != cudaSuccess) {
        cudaGetLastError();
        S->inv = nullptr;
        return LSQ_OK;
    }
    S->inv64 = !m32 || block_sweep_mode(S->nnz_M, n) == 1;
    const unsigned g = (unsigned)std::min<int64_t>(nblk, 1 << 20);
    if (m32) {
        LSQ_CUDA(cudaFuncSetAttribute(k_block_inverse<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SI_SMEM));
        k_block_inverse<float><<<g, SI_T, SI_SMEM, st>>>(n, S->mptr, S->mcol, S->mval32, S->mval, S->mdiag, S->inv, S->inv64);
    } else {
        LSQ_CUDA(cudaFuncSetAttribute(k_block_inverse<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SI_SMEM));
        k_block_inverse<double><<<g, SI_T, SI_SMEM, st>>>(n, S->mptr, S->mcol, S->mval, S->mval, S->mdiag, S->inv, 1);
    }
    count_launch();
    LSQ_CUDA(cudaGetLastError());
    return LSQ_OK;
}

lsq_status sb_levels(const SparseHandle* S, int64_t n, int* lev1_f, int* lev1_b, int* max_f, int* max_b,
                     unsigned* err, cudaStream_t st) {
    int res = 0;
    lsq_status r = resident_ctas((const void*)k_levels_blocked, SL_T, 0, &res);
    if (r != LSQ_OK) return r;
    const int64_t nblk = (n + SB_ROWS - 1) / SB_ROWS;
    unsigned grid = (unsigned)std::min<int64_t>(2 * nblk, res) & ~1u;
    int64_t nn = n;
    const int64_t *mptr = S->mptr, *mdiag = S->mdiag;
    const int32_t* mcol = S->mcol;
    unsigned max_polls = dep_wait_polls();
    void* params[] = {&nn, (void*)&mptr, (void*)&mcol, (void*)&mdiag, &lev1_f, &lev1_b, &max_f, &max_b, &err, &max_polls};
    LSQ_CUDA(cudaLaunchCooperativeKernel((const void*)k_levels_blocked, dim3(grid), dim3(SL_T), params, 0, st));
    count_launch();
    return LSQ_OK;
}

}  // namespace lsq
