// The band kernel per storage mode and rounding.
#include "dmrt.h"
#include "step_band.cuh"

namespace dmrt {

const void* band_kernel(int storage, int rounding) {
    using Mixed = Split<__half, float>;
    const bool sr = rounding == DMRT_ROUND_STOCHASTIC;
    switch (storage) {
        case DMRT_FP32: return (const void*)step_band_kernel<OneType<float>, false>;
        case DMRT_FP16:
            return sr ? (const void*)step_band_kernel<OneType<__half>, true>
                      : (const void*)step_band_kernel<OneType<__half>, false>;
        case DMRT_BF16:
            return sr ? (const void*)step_band_kernel<OneType<__nv_bfloat16>, true>
                      : (const void*)step_band_kernel<OneType<__nv_bfloat16>, false>;
        case DMRT_MIXED:
            return sr ? (const void*)step_band_kernel<Mixed, true> : (const void*)step_band_kernel<Mixed, false>;
        case DMRT_THETA32:
            return sr ? (const void*)step_band_kernel<ThetaSplit, true>
                      : (const void*)step_band_kernel<ThetaSplit, false>;
    }
    return nullptr;
}

}  // namespace dmrt
