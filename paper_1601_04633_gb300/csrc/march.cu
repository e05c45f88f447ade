// The march kernel per storage mode, rounding and steps per launch.
#include "dmrt.h"
#include "step_march.cuh"

namespace dmrt {

template <typename L, bool SR, int MINB>
static MarchForm form(int steps) {
    return {steps == 2 ? (const void*)step_march_kernel<L, SR, 2, MINB>
                       : (const void*)step_march_kernel<L, SR, 3, 3>,
            MarchGeo<L>::kSmem, MarchGeo<L>::kCols, MarchGeo<L>::kBox};
}

MarchForm march_form(int storage, int rounding, int steps) {
    using Mixed = Split<__half, float>;
    const bool sr = rounding == DMRT_ROUND_STOCHASTIC;
    switch (storage) {
        case DMRT_FP32: return form<OneType<float>, false, 3>(steps);
        case DMRT_FP16: return sr ? form<OneType<__half>, true, 4>(steps) : form<OneType<__half>, false, 4>(steps);
        case DMRT_BF16:
            return sr ? form<OneType<__nv_bfloat16>, true, 4>(steps) : form<OneType<__nv_bfloat16>, false, 4>(steps);
        case DMRT_MIXED: return sr ? form<Mixed, true, 4>(steps) : form<Mixed, false, 4>(steps);
        case DMRT_THETA32: return sr ? form<ThetaSplit, true, 4>(steps) : form<ThetaSplit, false, 4>(steps);
    }
    return {nullptr, 0, 0, 0};
}

}  // namespace dmrt
