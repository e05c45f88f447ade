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

template <bool FIRST>
static __global__ void __launch_bounds__(32)
    march_wait_probe_kernel(const __grid_constant__ MarchMaps maps, const __grid_constant__ MarchArgs M,
                            const __grid_constant__ PairConsts K, int item, int row, unsigned long long limit_ns) {
    using L = OneType<float>;
    extern __shared__ __align__(1024) unsigned char smem_m[];
    const int lane = threadIdx.x;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem_m + MarchGeo<L>::kWarp);
    if (lane == 0) {
        for (int s = 0; s < kMarchStages; ++s) mbar_init(&bars[s], s == row ? 2 : 1);
        mbar_fence_init();
    }
    __syncwarp();
    march_item<L, false, 3, FIRST>(maps.ld, maps.st, M, K.r, K.n, item, lane, smem_m, bars, limit_ns);
}

cudaError_t launch_march_wait_probe(const MarchMaps& maps, const MarchArgs& M, const PairConsts& K, int item, int row,
                                    bool first, unsigned long long limit_ns, cudaStream_t stream) {
    constexpr unsigned smem = MarchGeo<OneType<float>>::kSmem;
    const auto kernel = first ? march_wait_probe_kernel<true> : march_wait_probe_kernel<false>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<1, 32, smem, stream>>>(maps, M, K, item, row, limit_ns);
    return cudaGetLastError();
}

}  // namespace dmrt
