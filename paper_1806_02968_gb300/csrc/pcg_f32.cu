// FP32-value instantiations of the persistent PCG kernel (FP32 products and accumulation
// in the fused pass; FP64 vectors, dots and scalars; true residuals from FP64 values when
// an FP64 copy is supplied).
#include "pcg_launch.cuh"

namespace lsq {

template <int DTR, typename OPT>
static lsq_status f32_by_n(int64_t nmax, PcgArgs& a, int cap, cudaStream_t st) {
    switch (nmax) {
        case 128: return launch_pcg_one<LSQ_F32, DTR, 128, OPT>(a, cap, st);
        case 256: return launch_pcg_one<LSQ_F32, DTR, 256, OPT>(a, cap, st);
        case 512: return launch_pcg_one<LSQ_F32, DTR, 512, OPT>(a, cap, st);
        case 1024: return launch_pcg_one<LSQ_F32, DTR, 1024, OPT>(a, cap, st);
        case 2048:
            if (DTR == LSQ_F32) return launch_pcg_one<LSQ_F32, LSQ_F32, 2048, OPT>(a, cap, st);
            break;
    }
    set_error("FP32 dense PCG supports n <= 2048 (n <= 1024 with FP64 residuals)");
    return LSQ_ERR_UNSUPPORTED;
}

lsq_status launch_pcg_f32(int64_t nmax, int dtr, int opt_dtype, PcgArgs& a, int cap, cudaStream_t st) {
    if (dtr == LSQ_F64)
        return opt_dtype == LSQ_F32 ? f32_by_n<LSQ_F64, float>(nmax, a, cap, st)
                                    : f32_by_n<LSQ_F64, double>(nmax, a, cap, st);
    return opt_dtype == LSQ_F32 ? f32_by_n<LSQ_F32, float>(nmax, a, cap, st)
                                : f32_by_n<LSQ_F32, double>(nmax, a, cap, st);
}

}  // namespace lsq
