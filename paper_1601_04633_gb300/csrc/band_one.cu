// The band kernel across the GPU, one pair per thread, per storage mode and rounding.
#include "dmrt.h"
#include "step_band.cuh"

namespace dmrt {

template <typename L, bool SR>
static const void* form() {
    return (const void*)step_band_kernel<L, SR, false, true, kBandThreads>;
}

const void* band_one_kernel(int storage, int rounding) {
    using Mixed = Split<__half, float>;
    const bool sr = rounding == DMRT_ROUND_STOCHASTIC;
    switch (storage) {
        case DMRT_FP32: return form<OneType<float>, false>();
        case DMRT_FP16: return sr ? form<OneType<__half>, true>() : form<OneType<__half>, false>();
        case DMRT_BF16: return sr ? form<OneType<__nv_bfloat16>, true>() : form<OneType<__nv_bfloat16>, false>();
        case DMRT_MIXED: return sr ? form<Mixed, true>() : form<Mixed, false>();
        case DMRT_THETA32: return sr ? form<ThetaSplit, true>() : form<ThetaSplit, false>();
    }
    return nullptr;
}

}  // namespace dmrt
