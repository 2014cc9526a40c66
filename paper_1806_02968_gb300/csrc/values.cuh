// Scalar loads of matrix values as FP64 (exact for F64/F32/BF16; RN(hi + lo) for F32X2).
#pragma once
#include "common.cuh"

namespace lsq {

// A float as the same double, by integer operations alone: GB300 converts to and from 64-bit types
// (and does every other FP64 operation) at 2 lanes a clock and SM, integers at 64.
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), mag = u & 0x7fffffffu, ex = mag >> 23;
    unsigned hi = (mag >> 3) + 0x38000000u, lo = u << 29;    // normal: rebias the exponent
    if (ex - 1u >= 254u) {
        if (ex == 255u) {
            hi = (mag >> 3) + 0x70000000u;                   // infinity, NaN
        } else if (mag == 0u) {
            hi = lo = 0u;
        } else {                                             // subnormal: a normal double
            const int sh = __clz((int)mag) - 8;
            const unsigned m = mag << sh;
            hi = ((unsigned)(897 - sh) << 20) | ((m & 0x7fffffu) >> 3);
            lo = m << 29;
        }
    }
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)lo);
}

template <int DT> struct Val;   // load() widens by integer operations
template <> struct Val<LSQ_F64> {
    typedef double T;
    static __device__ __forceinline__ double load(const void* p, int64_t e) {
        return reinterpret_cast<const double*>(p)[e];
    }
};
template <> struct Val<LSQ_F32> {
    typedef float T;
    static __device__ __forceinline__ double load(const void* p, int64_t e) {
        return widen(reinterpret_cast<const float*>(p)[e]);
    }
};
template <> struct Val<LSQ_BF16> {
    typedef __nv_bfloat16 T;
    static __device__ __forceinline__ double load(const void* p, int64_t e) {
        return widen(__bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[e]));
    }
};
template <> struct Val<LSQ_F32X2> {
    static __device__ __forceinline__ double load(const void* p, int64_t e) {
        const float* f = reinterpret_cast<const float*>(p);
        return __dadd_rn((double)f[2 * e], (double)f[2 * e + 1]);
    }
};

// an FP32 or BF16 value as FP32
template <int DT>
__device__ __forceinline__ float load_f32(const void* p, int64_t e) {
    if constexpr (DT == LSQ_BF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[e]);
    else return reinterpret_cast<const float*>(p)[e];
}
// a value as FP64 by the hardware's conversion, for a pass that waits on memory and has FP64 slots
// to spare (CSR, one column: 0.162 ms per column pass of 3.2e7 entries, 0.190 ms with integer widening)
template <int DT>
__device__ __forceinline__ double load_f64(const void* p, int64_t e) {
    if constexpr (DT == LSQ_F32 || DT == LSQ_BF16) return (double)load_f32<DT>(p, e);
    else return Val<DT>::load(p, e);
}

}  // namespace lsq
