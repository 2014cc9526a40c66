// Cooperative launch of one k_pcg_dense instantiation (included by pcg_f64.cu / pcg_f32.cu).
#pragma once
#include "pcg_kernel.cuh"

namespace lsq {

constexpr int PCG_THREADS = 512;

template <int DT, int DTR, int NMAX, typename OPT>
lsq_status launch_pcg_one(PcgArgs& a, int grid_cap, cudaStream_t st) {
    auto kern = k_pcg_dense<DT, DTR, NMAX, OPT>;
    const size_t smem = pcg_smem_bytes(NMAX);
    LSQ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int dev = 0, sms = 0, per_sm = 0;
    LSQ_CUDA(cudaGetDevice(&dev));
    LSQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    LSQ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, PCG_THREADS, smem));
    if (per_sm < 1) { set_error("PCG kernel does not fit on an SM"); return LSQ_ERR_CUDA; }
    int T = sms;                   // one CTA per SM (the ring takes most of its shared memory)
    if (grid_cap > 0 && T > grid_cap) T = grid_cap;
    int64_t by_rows = a.m / 16;    // at least ~16 rows per CTA
    if (by_rows < 1) by_rows = 1;
    // Up to 16 columns side by side, the same number in every round, as long as a column on its group
    // alone takes no more time than the chip's latencies: when the others are done (or zero) it keeps its
    // group, no more.  A pass over a matrix of L2's size takes about as long as the barriers and vector
    // phases of an iteration, so the groups' copies of it together may have that size, and twice that from 8
    // columns on for the other types, whose passes are not bound by FP64 operations.  Larger matrices gain
    // little: 262,144 x 512 FP32, 4 columns 13.1 ms side by side, 14.3 ms one after the other, but 13.1
    // against 4.5 ms when three of them are zero.  60,001 x 201 FP32 (49 MB), 8 columns: 3.2 ms in eight
    // groups, 3.5 ms in four, 7 ms in one; one of 8 not zero: 3.2, 1.8 and 1.7 ms.
    const int64_t bytes = a.m * a.ld * (int64_t)elem_size(DT);
    const int64_t room = (int64_t)128 << (a.ncol >= 8 && DT != LSQ_F64 ? 21 : 20);
    int64_t most = T < 16 ? T : 16;
    if (most > room / bytes) most = room / bytes > 1 ? room / bytes : 1;
    const int64_t rounds = (a.ncol + most - 1) / most;
    a.NG = (int)((a.ncol + rounds - 1) / rounds);
    a.G = (int)(T / a.NG < by_rows ? T / a.NG : by_rows);
    const int G = a.G * a.NG;
    void* params[] = {&a};
    LSQ_CUDA(cudaLaunchCooperativeKernel((const void*)kern, dim3(G), dim3(PCG_THREADS), params, smem, st));
    count_launch();
    return LSQ_OK;
}

// Upper bound on the grid any instantiation may use (workspace sizing).
inline int pcg_max_grid() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

lsq_status launch_pcg_f64(int64_t nmax, int opt_dtype, PcgArgs& a, int cap, cudaStream_t st);
lsq_status launch_pcg_f32(int64_t nmax, int dtr, int opt_dtype, PcgArgs& a, int cap, cudaStream_t st);
lsq_status launch_pcg_f32x2(int64_t nmax, int dtr, int opt_dtype, PcgArgs& a, int cap, cudaStream_t st);
lsq_status launch_pcg_bf16(int64_t nmax, int dtr, int opt_dtype, PcgArgs& a, int cap, cudaStream_t st);

}  // namespace lsq
