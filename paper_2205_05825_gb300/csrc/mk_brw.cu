// Warp-level blind rotation (mk_bootstrap_warp.cuh): instantiation and launch.
#include "mk_bootstrap_warp.cuh"

namespace mk {
namespace {
// Gates per CTA for this batch: as many as spread the batch over the SMs,
// capped by the launch bound and by shared memory.
uint32_t warp_gates(uint32_t k, uint32_t n, uint32_t count, uint32_t sms) {
    uint32_t g = (count + sms - 1) / sms;
    if (g > (uint32_t)br::kWarpMaxGates) g = (uint32_t)br::kWarpMaxGates;
    while (g > 0 && br::warp_layout(k, n, g).total > kWarpSmemMax) --g;
    return g;
}
}  // namespace

bool warp_form_supported(const LaunchShape &S) {
    return S.form == MK_FORM_NTT2 && S.logN == 10 && S.d == 3 && S.bg_bit == 8 &&
           br::warp_layout(S.k, S.n, 1).total <= kWarpSmemMax;
}

cudaError_t launch_bootstrap_warp(const LaunchShape &S, const DeviceKeys &K, const GateDesc *desc,
                                  const uint32_t *ct_a, const uint32_t *ct_b, const uint32_t *abar_in,
                                  int64_t max_steps, uint32_t *ext, uint32_t *acc_out, uint32_t count,
                                  cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    if (!warp_form_supported(S) || K.tw_warp == nullptr) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const uint32_t g = warp_gates(S.k, S.n, count, (uint32_t)sms);
    const size_t smem = br::warp_layout(S.k, S.n, g).total;
    auto kern = br::bootstrap_warp_kernel;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const uint32_t grid = count < (uint32_t)sms ? count : (uint32_t)sms;
    kern<<<grid, 128 * g, smem, st>>>(S, K, desc, ct_a, ct_b, abar_in, max_steps, ext, acc_out, count);
    return cudaGetLastError();
}
}  // namespace mk
