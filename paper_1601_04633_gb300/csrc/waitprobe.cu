// dmrt_probe_bounded_wait: exercises the failure path of the step kernels'
// bounded device-side waits without faulting or hanging the GPU. One thread
// waits, through the same routine the step kernels use (mbar_wait_bounded), on
// an mbarrier that nothing ever completes; the wait must give up after the
// limit and report it, leaving the context usable.
#include <cuda_runtime.h>

#include <cstdio>

#include "dmrt.h"
#include "step_band.cuh"

void dmrt_internal_set_error(const char* msg);

namespace {

void set_error(const char* name, const char* what) {
    char msg[128];
    std::snprintf(msg, sizeof msg, "%s: %s", name, what);
    dmrt_internal_set_error(msg);
}

// [0]: 1 if the wait completed (it must not), 2 if it gave up; [1]: waited ns.
__device__ unsigned long long g_probe[2];

__global__ void wait_probe_kernel(unsigned long long limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    dmrt::mbar_init(&bar, 1);
    dmrt::mbar_fence_init();
    const unsigned long long t0 = dmrt::global_ns();
    const bool done = dmrt::mbar_wait_bounded(&bar, 0u, limit_ns);  // phase 0 never completes
    g_probe[0] = done ? 1ull : 2ull;
    g_probe[1] = dmrt::global_ns() - t0;
}

// Words of a message that carry no step's tag.
constexpr int kProbeWords = 8;  // per plane: columns 0 and 1 with two words on each side, rounded up
__device__ __align__(16) unsigned long long g_words[4 * kProbeWords];

__global__ void band_wait_probe_kernel(int kind, unsigned long long limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    dmrt::mbar_init(&bar, 1);
    dmrt::mbar_fence_init();
    const unsigned long long t0 = dmrt::global_ns();
    dmrt::F2 v[4];
    const bool done = kind == 0 ? dmrt::mail_read<1>(g_words + 2, kProbeWords, 0, false, false, 1u, v, limit_ns)
                                : dmrt::cluster_wait(&bar, 0u, limit_ns);
    g_probe[0] = done ? 1ull : 2ull;
    g_probe[1] = dmrt::global_ns() - t0;
}

int run_probe(const char* name, int kind, int64_t limit_ns, void* stream, int64_t* waited_ns) {
    if (limit_ns < 1000000 || limit_ns > (int64_t)dmrt::kWaitLimitNs || kind > 1) {
        set_error(name, "limit must be in [1 ms, 2 s], kind 0 or 1");
        return DMRT_E_ARG;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned long long out[2] = {0, 0};
    if (kind < 0) wait_probe_kernel<<<1, 32, 0, s>>>((unsigned long long)limit_ns);
    else band_wait_probe_kernel<<<1, 32, 0, s>>>(kind, (unsigned long long)limit_ns);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbolAsync(out, g_probe, sizeof out, 0, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        dmrt_internal_set_error(cudaGetErrorString(e));
        return DMRT_E_CUDA;
    }
    if (waited_ns) *waited_ns = (int64_t)out[1];
    if (out[0] == 2) {
        set_error(name, "the wait gave up after its limit, as designed");
        return DMRT_E_TIMEOUT;
    }
    set_error(name, "the wait completed although nothing arrived");
    return DMRT_OK;
}

}  // namespace

extern "C" int dmrt_probe_bounded_wait(int64_t limit_ns, void* stream, int64_t* waited_ns) {
    return run_probe("dmrt_probe_bounded_wait", -1, limit_ns, stream, waited_ns);
}

extern "C" int dmrt_probe_band_wait(int32_t kind, int64_t limit_ns, void* stream, int64_t* waited_ns) {
    return run_probe("dmrt_probe_band_wait", kind < 0 ? 2 : kind, limit_ns, stream, waited_ns);
}
