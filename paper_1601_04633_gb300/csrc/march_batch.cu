// The batched march kernel: float32 and mixed storage, by steps per launch.
#include "dmrt.h"
#include "step_march.cuh"

namespace dmrt {

template <typename L, bool SR, int MINB>
static MarchForm form(int steps) {
    return {steps == 2 ? (const void*)batch_march_kernel<L, SR, 2, MINB>
                       : (const void*)batch_march_kernel<L, SR, 3, 3>,
            MarchGeo<L>::kSmem, MarchGeo<L>::kCols, MarchGeo<L>::kBox};
}

MarchForm batch_march_form(int storage, int rounding, int steps) {
    using Mixed = Split<__half, float>;
    if (storage == DMRT_FP32) return form<OneType<float>, false, 3>(steps);
    if (storage == DMRT_MIXED)
        return rounding == DMRT_ROUND_STOCHASTIC ? form<Mixed, true, 4>(steps) : form<Mixed, false, 4>(steps);
    return {nullptr, 0, 0, 0};
}

}  // namespace dmrt
