// Sec. 3.3 and Alg. 3 for dense matrices.
//
// M = X^T X with x_tj = a_{i_t j} / d_j / sqrt(s p_t) is a contraction over the draws, and GB300
// multiplies FP64 at two FMAs a clock and SM: 12,777 draws of 512 columns took 4.0 ms there. It
// runs on the tensor cores instead, in the manner of Ozaki, Ogita, Oishi & Rump
// ("Error-free transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 59, 2012): every column is scaled by a power of two and
// cut into seven signed 8-bit digits, x = 2^e sum_p q_p 2^(-7-8p), which BF16 holds exactly; the
// products of digits p and q with p + q <= 7 are summed by bf16 MMAs with FP32 accumulators.
// Digits are at most 128, so a sum of 128 rows over the at most seven pairs of one p + q stays
// below 2^24 and is exact; it is then moved to 64-bit integers.  (The pairs with p + q = 7 join
// the last sum scaled by 2^-8, with its rounding.)  What remains are the digits' end at 2^-56 of a
// column's largest entry and the products that are left out, 2^-64 of the two largest: errors
// against sqrt(M_jj M_kk).  An entry whose terms are all far below that (a column with one entry that
// stands out) would keep fewer bits than an FP64 product gives it, so every entry's error is
// bounded beside the products, and the tiles with one that may pass 8 roundings of its terms are
// summed in FP64 (k_wide_check, k_wide_tiles).
// 12,777 draws of 512 columns: 0.40 ms (0.37 without the magnitudes), 0.12 ms for the digits and 0.02
// for the bound; in FP64 4.0 ms.  Error of M against extended precision (Frobenius, relative; FP64
// product in brackets): Gaussian 1.45e-16 (1.83e-16), 2 % heavy rows 1.44e-16 (1.88e-16), the same
// under uniform draws 1.75e-16 (2.95e-16), UDV 1.49e-16 (1.93e-16), FP32 values 1.42e-16
// (2.32e-16), semi-Gaussian 1.82e-16 (2.57e-16).
#include "dense_build.cuh"
#include "values.cuh"

#include <algorithm>

namespace lsq {

constexpr int OZ_P = 7;           // digits
constexpr int OZ_PL = OZ_P + 1;   // planes: the digits, and the magnitudes
constexpr int OZ_TILE = 64;       // columns of M per tile edge
constexpr int OZ_KC = 16;         // draws per stage
constexpr int OZ_STAGES = 4;
constexpr int OZ_FLUSH = 128;     // draws whose sums stay exact in FP32
constexpr int OZ_PITCH = OZ_TILE + 8;   // bf16 per staged row (16 bytes of padding: distinct banks)
constexpr int OZ_T = 256;
constexpr size_t OZ_STAGE = (size_t)2 * OZ_PL * OZ_KC * OZ_PITCH * 2;
constexpr int OZ_BAD = 1 << 20;   // exponent of a column with a non-finite entry

// sqrt(gamma_t), gamma_t = 1 / (s p_t), as a head and a tail: its square is gamma_t to far below
// the digits, so the roots add no error of their own to the sums (under the uniform density
// every draw has the same gamma, and the rounding of one root would shift all of M)
__global__ void k_oz_weight(const double* p, int64_t s, double2* rg) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < s; t += (int64_t)gridDim.x * blockDim.x) {
        const double g = __drcp_rn(__dmul_rn((double)s, p[t]));
        const double h = __dsqrt_rn(g);
        rg[t] = make_double2(h, __ddiv_rn(fma(-h, h, g), 2.0 * h));
    }
}
template <int DT>
__device__ __forceinline__ double oz_a(const lsq_matrix& A, int64_t row, int64_t j, double dj) {
    return __dmul_rn(Val<DT>::load(A.vals, row * A.ld + j), dj);
}
// largest |x_tj| of every column (bit patterns), 32 draws per block
template <int DT>
__global__ void __launch_bounds__(256) k_oz_max(lsq_matrix A, const int32_t* idx, const double2* rg, const double* inv_d,
                                                int64_t s, unsigned long long* mx) {
    const int64_t t0 = (int64_t)blockIdx.x * 32, t1 = min(s, t0 + 32);
    for (int64_t j = threadIdx.x; j < A.n; j += blockDim.x) {
        const double dj = inv_d[j];
        unsigned long long best = 0;
#pragma unroll 8
        for (int64_t t = t0; t < t1; ++t) {
            const unsigned long long b =
                (unsigned long long)__double_as_longlong(__dmul_rn(oz_a<DT>(A, idx[t], j, dj), rg[t].x)) & 0x7fffffffffffffffull;
            best = b > best ? b : best;
        }
        if (best) atomicMax(&mx[j], best);
    }
}
// e_j with |x_tj| < 2^e_j (x the product with the head, correctly rounded), and 1 / d_j scaled
// so that the digits' integer is a_ij times it times the root.  A column without a non-zero draw
// has the scale 0, so that all its digits are zero; e_j is no smaller than what keeps the scale finite.
__global__ void k_oz_exp(const unsigned long long* mx, const double* inv_d, int64_t n, int* e, double* sd) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int ex = (int)(mx[j] >> 52);
    int ej = ex == 0x7ff ? OZ_BAD : 0;
    double sj = 0.0;
    if (mx[j] != 0 && ej != OZ_BAD) {
        ej = max(max(ex, 1) - 1022, ilogb(inv_d[j]) + 55 - 1022);
        sj = scalbn(inv_d[j], 55 - ej);
    }
    e[j] = ej;
    sd[j] = sj;
}
// Digits of the integer nearest x0 + x1, |x0| < 2^55, x1 the rounding error of x0.  Integer
// arithmetic on the bits: FP64 operations and conversions run at 1/64 of the integer rate.
__device__ __forceinline__ void oz_digits(double x0, double x1, int (&d)[OZ_P]) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x0);
    const int ex = (int)((b >> 52) & 0x7ff);
    const unsigned long long m = (b & ((1ull << 52) - 1)) | (ex ? 1ull << 52 : 0ull);
    const int sh = max(ex, 1) - 1075;             // |x0| = m 2^sh, sh <= 2
    long long y;
    if (sh >= 0) y = (long long)(m << min(sh, 2));
    else y = sh > -55 ? (long long)((m + (1ull << (-sh - 1))) >> -sh) : 0;
    if (b >> 63) y = -y;
    // the tail is worth a unit only where a unit of x0 is one or more: at most two
    if (sh >= 0) y += (int)__double2loint(__dadd_rn(x1, 0x1.8p52));
#pragma unroll
    for (int p = OZ_P - 1; p > 0; --p) {
        d[p] = (int)(signed char)(y & 0xff);
        y = (y - d[p]) >> 8;
    }
    d[0] = (int)y;                                // |d_0| <= 128
}
// |x0| 2^-55 cut to a bf16, from below; a non-zero one at least 2^-60, so that products stay normal
__device__ __forceinline__ unsigned oz_magnitude(double x0) {
    const unsigned hi = (unsigned)__double2hiint(x0) & 0x7fffffffu;
    if (hi == 0u && __double2loint(x0) == 0) return 0u;
    const int b = (int)(hi >> 13) - ((1023 + 55 - 127) << 7);   // rebias the exponent, keep 7 bits
    return (unsigned)max(b, (127 - 60) << 7);
}
__device__ __forceinline__ unsigned bf16_of_int(int v) { return __float_as_uint((float)v) >> 16; }
template <int DT>
__device__ __forceinline__ void oz_entry(const lsq_matrix& A, int64_t row, int64_t j, double sd, double2 g,
                                         int (&d)[OZ_P], unsigned& mag) {
    const double t = oz_a<DT>(A, row, j, sd);
    const double x0 = __dmul_rn(t, g.x);
    oz_digits(x0, fma(t, g.y, fma(t, g.x, -x0)), d);
    mag = oz_magnitude(x0);
}
// digits and magnitudes of draws [t0, t0 + rows) (zero beyond s and n): q[p][t - t0][j], two
// columns a thread
template <int DT>
__global__ void __launch_bounds__(256) k_oz_slice(lsq_matrix A, const int32_t* idx, const double2* rg,
                                                  const double* sd, const int* e, int64_t s, int64_t t0,
                                                  int64_t rows, int npad, unsigned* q) {
    const int half = npad >> 1;
    const int64_t plane = rows * half;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < plane; w += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = w / half, t = t0 + r;
        const int j = 2 * (int)(w - r * half);
        int d0[OZ_P] = {}, d1[OZ_P] = {};
        unsigned m0 = 0, m1 = 0;
        if (t < s) {
            const int64_t row = idx[t];
            const double2 g = rg[t];
            if (j < A.n && e[j] != OZ_BAD) oz_entry<DT>(A, row, j, sd[j], g, d0, m0);
            if (j + 1 < A.n && e[j + 1] != OZ_BAD) oz_entry<DT>(A, row, j + 1, sd[j + 1], g, d1, m1);
        }
#pragma unroll
        for (int p = 0; p < OZ_P; ++p) q[p * plane + w] = bf16_of_int(d0[p]) | (bf16_of_int(d1[p]) << 16);
        q[OZ_P * plane + w] = m0 | (m1 << 16);
    }
}

__device__ __forceinline__ void ldsm4t(unsigned (&r)[4], const void* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// both halves times 2^-8 (exact)
__device__ __forceinline__ unsigned bf16x2_scale(unsigned v) {
    unsigned r;
    asm("mul.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0x3b803b80u));
    return r;
}

// part[z][i][j] (+)= sum over split z's draws of x_ti x_tj for tile pair (ti <= tj).  8 warps: 4
// row groups of 16 by 2 column groups of 32; every warp keeps one FP32 accumulator tile per
// p + q and moves it to its 64-bit totals every 128 draws.  Digits arrive by cp.async in four
// stages of 16 draws.  mag[z][i][j] (+)= the same sums of the magnitudes, a lower bound of sum |x_ti| |x_tj|
// in units of 2^(e_i + e_j).  Bound: MMA issue (35 MMAs per 16 x 8 x 16 block of M).
__global__ void __launch_bounds__(OZ_T, 1) k_oz_gemm(const unsigned short* q, int64_t rows, int npad, int64_t n,
                                                     const int* e, int64_t per_split, int ntile, double* part,
                                                     float* mag, int accumulate) {
    extern __shared__ __align__(16) unsigned char oz_smem[];
    int ti = 0, rest = blockIdx.x;
    while (rest >= ntile - ti) { rest -= ntile - ti; ++ti; }
    const int tj = ti + rest;
    const int64_t r0 = (int64_t)blockIdx.y * per_split, r1 = min(rows, r0 + per_split);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int wi = (wid >> 1) * 16, wj = (wid & 1) * 32;
    const int nst = r1 > r0 ? (int)((r1 - r0) / OZ_KC) : 0;   // rows is a multiple of 128
    auto stage = [&](int k) {
        unsigned char* dst = oz_smem + (size_t)(k % OZ_STAGES) * OZ_STAGE;
        const int64_t t = r0 + (int64_t)k * OZ_KC;
        // 2 operands x 8 planes x 16 rows x 8 chunks of 16 bytes
        for (int c = tid; c < 2 * OZ_PL * OZ_KC * 8; c += OZ_T) {
            const int ch = c & 7, r = (c >> 3) & (OZ_KC - 1), pl = c >> 7;    // plane index 0..15
            const int side = pl >= OZ_PL ? 1 : 0, p = pl - side * OZ_PL;
            const unsigned short* src = q + ((int64_t)p * rows + t + r) * npad + (side ? tj : ti) * OZ_TILE + ch * 8;
            const unsigned s = (unsigned)__cvta_generic_to_shared(dst + ((size_t)(pl * OZ_KC + r) * OZ_PITCH + ch * 8) * 2);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(src) : "memory");
        }
    };
    float acc[OZ_P][4][4], macc[4][4];
    long long hi[4][4], lo[4][4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            hi[nt][v] = 0; lo[nt][v] = 0; macc[nt][v] = 0.f;
#pragma unroll
            for (int d = 0; d < OZ_P; ++d) acc[d][nt][v] = 0.f;
        }
    for (int k = 0; k < OZ_STAGES - 1; ++k) {
        if (k < nst) stage(k);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int k = 0; k < nst; ++k) {
        asm volatile("cp.async.wait_group %0;" ::"n"(OZ_STAGES - 2) : "memory");
        __syncthreads();   // stage k is here for every warp, and stage k - 1 is free
        if (k + OZ_STAGES - 1 < nst) stage(k + OZ_STAGES - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const unsigned short* S = reinterpret_cast<const unsigned short*>(oz_smem + (size_t)(k % OZ_STAGES) * OZ_STAGE);
        const int mid = lane >> 3, mr = lane & 7;
        unsigned a[OZ_P][4];
#pragma unroll
        for (int p = 0; p < OZ_P; ++p)
            ldsm4t(a[p], S + (size_t)(p * OZ_KC + (mid >> 1) * 8 + mr) * OZ_PITCH + wi + (mid & 1) * 8);
#pragma unroll
        for (int jp = 0; jp < 2; ++jp) {
#pragma unroll
            for (int qq = 0; qq < OZ_P; ++qq) {
                unsigned b[4];
                ldsm4t(b, S + (size_t)((OZ_PL + qq) * OZ_KC + (mid & 1) * 8 + mr) * OZ_PITCH + wj + jp * 16 + (mid >> 1) * 8);
#pragma unroll
                for (int p = 0; p + qq < OZ_P; ++p) {
                    mma_bf16(acc[p + qq][2 * jp], a[p], b[0], b[1]);
                    mma_bf16(acc[p + qq][2 * jp + 1], a[p], b[2], b[3]);
                }
                if (qq > 0) {   // p + q = 7, scaled by 2^-8 into the sum of p + q = 6
#pragma unroll
                    for (int v = 0; v < 4; ++v) b[v] = bf16x2_scale(b[v]);
                    mma_bf16(acc[OZ_P - 1][2 * jp], a[OZ_P - qq], b[0], b[1]);
                    mma_bf16(acc[OZ_P - 1][2 * jp + 1], a[OZ_P - qq], b[2], b[3]);
                }
            }
        }
        ldsm4t(a[0], S + (size_t)(OZ_P * OZ_KC + (mid >> 1) * 8 + mr) * OZ_PITCH + wi + (mid & 1) * 8);
#pragma unroll
        for (int jp = 0; jp < 2; ++jp) {
            unsigned b[4];
            ldsm4t(b, S + (size_t)((OZ_PL + OZ_P) * OZ_KC + (mid & 1) * 8 + mr) * OZ_PITCH + wj + jp * 16 + (mid >> 1) * 8);
            mma_bf16(macc[2 * jp], a[0], b[0], b[1]);
            mma_bf16(macc[2 * jp + 1], a[0], b[2], b[3]);
        }
        if ((k + 1) % (OZ_FLUSH / OZ_KC) == 0 || k + 1 == nst) {
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    int d[OZ_P];
#pragma unroll
                    for (int x = 0; x < OZ_P; ++x) { d[x] = __float2int_rn(acc[x][nt][v]); acc[x][nt][v] = 0.f; }
                    hi[nt][v] += ((long long)d[0] << 16) + ((long long)d[1] << 8) + d[2];
                    lo[nt][v] += ((long long)d[3] << 24) + ((long long)d[4] << 16) + ((long long)d[5] << 8) + d[6];
                }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    double* out = part + (int64_t)blockIdx.y * n * n;
    float* mout = mag + (int64_t)blockIdx.y * n * n;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int64_t i = (int64_t)ti * OZ_TILE + wi + (lane >> 2) + (v >> 1) * 8;
            const int64_t j = (int64_t)tj * OZ_TILE + wj + nt * 8 + 2 * (lane & 3) + (v & 1);
            if (i < n && j < n) {
                double x = fma((double)lo[nt][v], 0x1p-48, (double)hi[nt][v] * 0x1p-16);
                const int ei = e[i], ej = e[j];
                if (ei == OZ_BAD || ej == OZ_BAD) x = __longlong_as_double(0x7ff8000000000000ll);
                else x = scalbn(x, ei + ej - 14);
                out[i * n + j] = accumulate ? out[i * n + j] + x : x;
                mout[i * n + j] = accumulate ? mout[i * n + j] + macc[nt][v] : macc[nt][v];
            }
        }
}

// Column sums of the magnitudes, rounded up to multiples of 2^-24 (whole numbers, so that the sum
// does not depend on the order), 64 draws per block.
__global__ void __launch_bounds__(256) k_oz_sums(const unsigned short* mag, int64_t rows, int npad, int64_t n,
                                                 unsigned long long* sum) {
    const int64_t t0 = (int64_t)blockIdx.x * 64, t1 = min(rows, t0 + 64);
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
        unsigned v = 0;
#pragma unroll 8
        for (int64_t t = t0; t < t1; ++t)
            v += (unsigned)__float2int_ru(__uint_as_float((unsigned)mag[t * npad + j] << 16) * 0x1p24f);
        if (v) atomicAdd(&sum[j], (unsigned long long)v);
    }
}
// Marks the tiles with an entry that the digits may leave less accurate than an FP64 product.  The
// digits' errors in entry (i, j) are at most 2^-56 (sum |x_ti| + sum |x_tj|) from the digits' end and
// 5 * 2^-64 a draw from the products left out, in units of 2^(e_i + e_j); an FP64 product rounds each term
// four times before it adds them.  Accepted: 2^-50 sum |x_ti| |x_tj|, eight roundings of the terms, if all of
// the digits' errors had one sign (they do not: where this bound is met the error measured is at most a
// fifth of the FP64 product's, Gaussian, UDV, heavy rows and semi-Gaussian at n = 40 to 512, and
// these meet it three times over).  No common draw: nothing to lose.  The magnitudes are cut to 8
// bits: the sums of one column are taken 2^-7 higher.
__global__ void k_wide_check(int64_t n, int64_t s, int splits, int ntile, const float* mag,
                             const unsigned long long* sum, const int* e, int* wide) {
    const int64_t total = n * n;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < total; w += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = w / n, j = w - i * n;
        if (j < i || e[i] == OZ_BAD || e[j] == OZ_BAD) continue;
        float b = 0.f;
        for (int z = 0; z < splits; ++z) b += mag[(int64_t)z * total + w];
        if (b == 0.f) continue;
        const float need = (1.f + 0x1p-6f) * 0x1p-24f * (float)(sum[i] + sum[j]) + 6 * 0x1p-8f * (float)s;
        if (need > 64.f * b) wide[(i / OZ_TILE) * ntile + j / OZ_TILE] = 1;
    }
}
// part[z][i][j] of a marked tile in FP64: 4 x 4 entries a thread, 16 draws at a time through shared
// memory.  Bound: FP64 FMAs, two a clock and SM (all tiles of 12,777 draws of 512 columns: 4.0 ms).
template <int DT>
__global__ void __launch_bounds__(256) k_wide_tiles(lsq_matrix A, const int32_t* idx, const double* p,
                                                    const double* inv_d, int64_t s, int64_t per_split, int ntile,
                                                    const int* wide, double* part) {
    int ti = 0, rest = blockIdx.x;
    while (rest >= ntile - ti) { rest -= ntile - ti; ++ti; }
    const int tj = ti + rest;
    if (!wide[ti * ntile + tj]) return;
    const int64_t n = A.n, i0 = (int64_t)ti * OZ_TILE, j0 = (int64_t)tj * OZ_TILE;
    const int64_t t_begin = min(s, (int64_t)blockIdx.y * per_split), t_end = min(s, t_begin + per_split);
    __shared__ double Xi[OZ_KC][OZ_TILE], Xj[OZ_KC][OZ_TILE];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc[4][4] = {};
    for (int64_t t0 = t_begin; t0 < t_end; t0 += OZ_KC) {
        for (int w = threadIdx.x; w < OZ_KC * OZ_TILE; w += 256) {
            const int tt = w / OZ_TILE, c = w % OZ_TILE;
            const int64_t t = t0 + tt;
            double vi = 0.0, vj = 0.0;
            if (t < t_end) {
                const int64_t row = idx[t];
                const double g = __drcp_rn(__dmul_rn((double)s, p[t]));
                if (i0 + c < n) vi = __dmul_rn(oz_a<DT>(A, row, i0 + c, inv_d[i0 + c]), g);
                if (j0 + c < n) vj = oz_a<DT>(A, row, j0 + c, inv_d[j0 + c]);
            }
            Xi[tt][c] = vi;
            Xj[tt][c] = vj;
        }
        __syncthreads();
#pragma unroll
        for (int tt = 0; tt < OZ_KC; ++tt) {
            double a[4], b[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) { a[r] = Xi[tt][ty * 4 + r]; b[r] = Xj[tt][tx * 4 + r]; }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[r][q] = fma(a[r], b[q], acc[r][q]);
        }
        __syncthreads();
    }
    double* out = part + (int64_t)blockIdx.y * n * n;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = i0 + ty * 4 + r, j = j0 + tx * 4 + q;
            if (i < n && j < n) out[i * n + j] = acc[r][q];
        }
}

// M[j][k] = M[k][j] = sum_z part[z][j][k] for j <= k (fixed order); zero diagonal -> 1.
__global__ void k_reduce_M(int64_t n, int splits, const double* part, double* M, unsigned long long* n_fixed) {
    int64_t total = n * n;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t j = e / n, k = e % n;
        if (k < j) continue;
        double v = 0.0;
        for (int z = 0; z < splits; ++z) v += part[(int64_t)z * total + e];
        if (j == k && v == 0.0) { v = 1.0; atomicAdd(n_fixed, 1ull); }
        M[j * n + k] = v;
        M[k * n + j] = v;
    }
}

template <int DT>
static lsq_status normal_matrix(const lsq_matrix* A, const int32_t* idx, const double* p, const double* inv_d,
                                int64_t s, double* M, unsigned long long* n_fixed, cudaStream_t st) {
    const int64_t n = A->n;
    const int ntile = (int)((n + OZ_TILE - 1) / OZ_TILE), npad = ntile * OZ_TILE;
    const int tiles = ntile * (ntile + 1) / 2;
    // draws per chunk, the same number in each: digits of at most 112 MB, which stay in L2 between the kernels
    const int64_t srows = (s + OZ_FLUSH - 1) / OZ_FLUSH * OZ_FLUSH;
    const int64_t most = std::max<int64_t>(((int64_t)112 << 20) / (2 * OZ_PL * npad) / OZ_FLUSH, 1);
    const int64_t chunks = (srows / OZ_FLUSH + most - 1) / most;
    const int64_t chunk = (srows / OZ_FLUSH + chunks - 1) / chunks * OZ_FLUSH;
    // about one CTA per SM: each split takes at least 128 draws of a chunk
    int64_t splits = std::max<int64_t>(152 / tiles, 1);
    splits = std::min(splits, chunk / OZ_FLUSH);
    const int64_t per = ((chunk + splits - 1) / splits + OZ_FLUSH - 1) / OZ_FLUSH * OZ_FLUSH;
    splits = (chunk + per - 1) / per;
    Scratch sc;
    auto r256 = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t o_rg = 0, o_mx = r256(16 * (size_t)s), o_e = o_mx + r256(8 * (size_t)n),
                 o_sd = o_e + r256(4 * (size_t)n), o_sum = o_sd + r256(8 * (size_t)n),
                 o_wide = o_sum + r256(8 * (size_t)n), o_q = o_wide + r256(4 * (size_t)ntile * ntile),
                 o_part = o_q + r256((size_t)2 * OZ_PL * chunk * npad),
                 o_mag = o_part + r256(8 * (size_t)splits * n * n), total = o_mag + 4 * (size_t)splits * n * n;
    LSQ_CUDA(sc.alloc(total, st));
    char* base = sc.as<char>();
    double2* rg = (double2*)(base + o_rg);
    double* sd = (double*)(base + o_sd);
    unsigned long long* mx = (unsigned long long*)(base + o_mx);
    int* e = (int*)(base + o_e);
    unsigned* q = (unsigned*)(base + o_q);
    double* part = (double*)(base + o_part);
    float* mag = (float*)(base + o_mag);
    unsigned long long* sum = (unsigned long long*)(base + o_sum);
    int* wide = (int*)(base + o_wide);
    LSQ_CUDA(cudaMemsetAsync(mx, 0, 8 * (size_t)n, st));
    LSQ_CUDA(cudaMemsetAsync(sum, 0, o_q - o_sum, st));   // and no tile marked
    k_oz_weight<<<(unsigned)std::min<int64_t>((s + 255) / 256, 4096), 256, 0, st>>>(p, s, rg);
    k_oz_max<DT><<<(unsigned)((s + 31) / 32), 256, 0, st>>>(*A, idx, rg, inv_d, s, mx);
    k_oz_exp<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(mx, inv_d, n, e, sd);
    count_launch(3);
    const size_t smem = OZ_STAGE * OZ_STAGES;
    LSQ_CUDA(cudaFuncSetAttribute(k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    for (int64_t t0 = 0; t0 < s; t0 += chunk) {
        const int64_t rows = std::min(chunk, srows - t0);
        const int64_t work = rows * (npad / 2);
        k_oz_slice<DT><<<(unsigned)std::min<int64_t>((work + 255) / 256, 152 * 32), 256, 0, st>>>(
            *A, idx, rg, sd, e, s, t0, rows, npad, q);
        // every split runs in every chunk (a split past the chunk's rows adds nothing)
        k_oz_gemm<<<dim3((unsigned)tiles, (unsigned)splits), OZ_T, smem, st>>>(
            reinterpret_cast<const unsigned short*>(q), rows, npad, n, e, per, ntile, part, mag, t0 > 0 ? 1 : 0);
        k_oz_sums<<<(unsigned)((rows + 63) / 64), 256, 0, st>>>(
            reinterpret_cast<const unsigned short*>(q) + OZ_P * rows * npad, rows, npad, n, sum);
        count_launch(3);
    }
    k_wide_check<<<(unsigned)std::min<int64_t>((n * n + 255) / 256, 152 * 16), 256, 0, st>>>(n, s, (int)splits, ntile, mag,
                                                                                            sum, e, wide);
    k_wide_tiles<DT><<<dim3((unsigned)tiles, (unsigned)splits), 256, 0, st>>>(
        *A, idx, p, inv_d, s, ((s + splits - 1) / splits + OZ_KC - 1) / OZ_KC * OZ_KC, ntile, wide, part);
    count_launch(2);
    k_reduce_M<<<(unsigned)std::min<int64_t>((n * n + 255) / 256, 152 * 16), 256, 0, st>>>(n, (int)splits, part, M, n_fixed);
    count_launch();
    LSQ_CUDA(cudaGetLastError());
    return LSQ_OK;
}

lsq_status dense_normal_matrix(const lsq_matrix* A, const int32_t* idx, const double* p, const double* inv_d,
                               int64_t s, double* M, unsigned long long* n_fixed, cudaStream_t st) {
    switch (A->dtype) {
        case LSQ_F64: return normal_matrix<LSQ_F64>(A, idx, p, inv_d, s, M, n_fixed, st);
        case LSQ_F32: return normal_matrix<LSQ_F32>(A, idx, p, inv_d, s, M, n_fixed, st);
        case LSQ_BF16: return normal_matrix<LSQ_BF16>(A, idx, p, inv_d, s, M, n_fixed, st);
        default: return normal_matrix<LSQ_F32X2>(A, idx, p, inv_d, s, M, n_fixed, st);
    }
}

// ---------------------------------------------------------------------------------------
// The SGS operator: column j is Alg. 3 on e_j, the t forward and t backward sweeps in the
// natural row order.  A CTA runs C columns together, 32 rows at a time: the warps split the sum
// over all other entries (lane = row, so M, symmetric, is read along its rows), and the 32 x 32
// triangle is solved by one product with its inverse.  All of the work is FP64 FMAs of full
// warps (a warp per column with a warp reduction per row, as before, spent its time in FP64
// shuffle-adds and divisions), so the kernel is bound by the FP64 pipe: (2t - 1/2) n^3 FMAs.
// n = 512, t = 1: 0.45 ms against 2.06 ms; n = 400, t = 5: 1.47 ms against 7.73 ms (0.98 ms of
// FMAs at the pipe's rate).
// C is the columns each SM gets when they are spread over all of them, up to 4.
// ---------------------------------------------------------------------------------------
constexpr int SG_T = 256, SG_W = SG_T / 32;

// inverses of the 32 x 32 lower diagonal blocks (the identity beyond n), a warp per block:
// lane j holds column j.  lt[b][k][r] = inv(r, k) (forward), lo[b][k][r] = inv(k, r) (backward,
// the upper block's inverse).
__global__ void __launch_bounds__(32) k_tri_inv32(int64_t n, const double* M, double* lt, double* lo) {
    __shared__ double L[32][33];
    const int lane = threadIdx.x;
    const int64_t k0 = (int64_t)blockIdx.x * 32;
    for (int r = 0; r < 32; ++r)
        L[r][lane] = (k0 + r < n && k0 + lane < n) ? M[(k0 + r) * n + k0 + lane] : (r == lane ? 1.0 : 0.0);
    __syncwarp();
    const double rd = 1.0 / L[lane][lane];
    double x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < i; ++k) t = fma(L[i][k], x[k], t);
        const double rdi = __shfl_sync(0xffffffffu, rd, i);   // every lane takes part
        const double rhs = i == lane ? 1.0 : 0.0;
        x[i] = i < lane ? 0.0 : (rhs - t) * rdi;
    }
    double* a = lt + (int64_t)blockIdx.x * 1024;
    double* b = lo + (int64_t)blockIdx.x * 1024;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        a[lane * 32 + i] = x[i];   // inv(i, lane)
        b[i * 32 + lane] = x[i];
    }
}

template <typename OT, int C>
__global__ void __launch_bounds__(SG_T) k_sgs_columns(int64_t n, int sweeps, const double* M, const double* lt,
                                                      const double* lo, OT* op) {
    extern __shared__ __align__(16) double sg_smem[];
    double* E = sg_smem;                        // n32 x C
    const int nb = (int)((n + 31) / 32);
    double* red = E + (size_t)nb * 32 * C;      // SG_W x 32 x C
    double* S = red + SG_W * 32 * C;            // 32 x C
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * C;
    constexpr int HS = SG_W / C;                // warps per column in the triangular product
    constexpr int KP = 32 / HS;                 // entries of a row each of them takes
    for (int t = tid; t < nb * 32 * C; t += SG_T) E[t] = 0.0;
    __syncthreads();
    const int b0 = (int)(j0 / 32);
    for (int sw = 0; sw < 2 * sweeps; ++sw) {
        const bool fwd = sw < sweeps, first = sw == 0;
        for (int kk = first ? b0 : 0; kk < nb; ++kk) {
            const int kb = fwd ? kk : nb - 1 - kk;
            const int64_t k0 = (int64_t)kb * 32, r = k0 + lane;
            // the inverse's entries this thread multiplies (loaded ahead of the long sum)
            double iv[KP];
            const double* ib = (fwd ? lt : lo) + (int64_t)kb * 1024;
            const int hs = w / C;
            if (w < C * HS) {
#pragma unroll
                for (int t = 0; t < KP; ++t) iv[t] = ib[(hs * KP + t) * 32 + lane];
            }
            // sum over all entries but the block's own triangle; on the first sweep only the
            // blocks from b0 on hold anything yet
            double acc[C];
#pragma unroll
            for (int c = 0; c < C; ++c) acc[c] = 0.0;
            const int64_t l0 = first ? (int64_t)b0 * 32 : 0, l1 = first ? k0 : n;
            const double* Mr = M + r;
            const bool rin = r < n;
#pragma unroll 8
            for (int64_t l = l0 + w; l < l1; l += SG_W) {
                double m = rin ? Mr[l * n] : 0.0;
                if (l >= k0 && l < k0 + 32 && (fwd ? l <= r : l >= r)) m = 0.0;
#pragma unroll
                for (int c = 0; c < C; ++c) acc[c] = fma(m, E[l * C + c], acc[c]);
            }
#pragma unroll
            for (int c = 0; c < C; ++c) red[(w * 32 + lane) * C + c] = acc[c];
            __syncthreads();
            if (tid < 32 * C) {
                const int rr = tid / C, c = tid % C;
                double s = 0.0;   // the small terms first, then the unit vector's entry
#pragma unroll
                for (int v = 0; v < SG_W; ++v) s += red[(v * 32 + rr) * C + c];
                S[tid] = (k0 + rr == j0 + c ? 1.0 : 0.0) - s;
            }
            __syncthreads();
            if (w < C * HS) {
                const int c = w % C;
                double x = 0.0;
#pragma unroll
                for (int t = 0; t < KP; ++t) x = fma(iv[t], S[(hs * KP + t) * C + c], x);
                red[(hs * C + c) * 32 + lane] = x;
            }
            __syncthreads();
            if (tid < 32 * C) {
                const int rr = tid / C, c = tid % C;
                double x = 0.0;
#pragma unroll
                for (int v = 0; v < HS; ++v) x += red[(v * C + c) * 32 + rr];
                E[(k0 + rr) * C + c] = x;
            }
            __syncthreads();
        }
    }
    for (int64_t t = tid; t < n * C; t += SG_T) {
        const int64_t k = t / C, c = t % C;
        if (j0 + c < n) op[k * n + j0 + c] = (OT)E[t];
    }
}

// Shared memory for n <= 2048 columns.  The limit is one for the whole process and set to the most,
// so that threads that build handles of different sizes do not lower it under one another.
constexpr size_t sg_bytes(int64_t n, int C) {
    return 8 * ((size_t)((n + 31) / 32) * 32 * C + SG_W * 32 * C + 32 * C);
}
template <typename OT, int C>
static lsq_status sgs_columns(int64_t n, int sweeps, const double* M, const double* lt, const double* lo, OT* op,
                              cudaStream_t st) {
    const size_t smem = sg_bytes(n, C);
    LSQ_CUDA(cudaFuncSetAttribute(k_sgs_columns<OT, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sg_bytes(2048, C)));
    k_sgs_columns<OT, C><<<(unsigned)((n + C - 1) / C), SG_T, smem, st>>>(n, sweeps, M, lt, lo, op);
    count_launch();
    LSQ_CUDA(cudaGetLastError());
    return LSQ_OK;
}
template <typename OT>
static lsq_status sgs_operator(int64_t n, int sweeps, const double* M, OT* op, cudaStream_t st) {
    const int64_t nb = (n + 31) / 32;
    Scratch sc;
    LSQ_CUDA(sc.alloc(16 * (size_t)nb * 1024, st));
    double* lt = sc.as<double>();
    double* lo = lt + nb * 1024;
    k_tri_inv32<<<(unsigned)nb, 32, 0, st>>>(n, M, lt, lo);
    count_launch();
    if (n <= 152) return sgs_columns<OT, 1>(n, sweeps, M, lt, lo, op, st);
    if (n <= 304) return sgs_columns<OT, 2>(n, sweeps, M, lt, lo, op, st);
    if (n <= 456) return sgs_columns<OT, 3>(n, sweeps, M, lt, lo, op, st);
    return sgs_columns<OT, 4>(n, sweeps, M, lt, lo, op, st);
}
lsq_status dense_sgs_operator(int64_t n, int sweeps, const double* M, void* op, int op_dtype, cudaStream_t st) {
    if (op_dtype == LSQ_F32) return sgs_operator<float>(n, sweeps, M, (float*)op, st);
    return sgs_operator<double>(n, sweeps, M, (double*)op, st);
}

}  // namespace lsq
