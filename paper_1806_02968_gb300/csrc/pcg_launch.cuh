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
    // up to 16 columns side by side, the same number in every round
    const int64_t most = T < 16 ? T : 16;
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
