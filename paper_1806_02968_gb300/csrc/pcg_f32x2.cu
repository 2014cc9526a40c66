// Double-float instantiations of the persistent PCG kernel: values stored as float pairs
// (hi, lo), products and sums in double-float on the FP32 units; FP64 vectors, dots and
// scalars; true residuals from FP64 values when an FP64 copy is supplied.
#include "pcg_launch.cuh"

namespace lsq {

template <int DTR, typename OPT>
static lsq_status x2_by_n(int64_t nmax, PcgArgs& a, int cap, cudaStream_t st) {
    switch (nmax) {
        case 128: return launch_pcg_one<LSQ_F32X2, DTR, 128, OPT>(a, cap, st);
        case 256: return launch_pcg_one<LSQ_F32X2, DTR, 256, OPT>(a, cap, st);
        case 512: return launch_pcg_one<LSQ_F32X2, DTR, 512, OPT>(a, cap, st);
        case 1024: return launch_pcg_one<LSQ_F32X2, DTR, 1024, OPT>(a, cap, st);
    }
    set_error("double-float dense PCG supports n <= 1024");
    return LSQ_ERR_UNSUPPORTED;
}

lsq_status launch_pcg_f32x2(int64_t nmax, int dtr, int opt_dtype, PcgArgs& a, int cap, cudaStream_t st) {
    if (dtr == LSQ_F64)
        return opt_dtype == LSQ_F32 ? x2_by_n<LSQ_F64, float>(nmax, a, cap, st)
                                    : x2_by_n<LSQ_F64, double>(nmax, a, cap, st);
    return opt_dtype == LSQ_F32 ? x2_by_n<LSQ_F32X2, float>(nmax, a, cap, st)
                                : x2_by_n<LSQ_F32X2, double>(nmax, a, cap, st);
}

}  // namespace lsq
