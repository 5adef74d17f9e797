// Warp, team, shared and N = 256 blind rotations (mk_bootstrap_warp.cuh, _team, _shared, _small):
// instantiation, launch, and which of them a launch gets.
#include "mk_bootstrap_shared.cuh"
#include "mk_bootstrap_small.cuh"
#include "mk_bootstrap_team.cuh"

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
    auto kern = S.skip_key_step < 0 ? br::bootstrap_warp_kernel<false> : br::bootstrap_warp_kernel<true>;
    e = br::allow_smem(kern);
    if (e != cudaSuccess) return e;
    const uint32_t grid = count < (uint32_t)sms ? count : (uint32_t)sms;
    kern<<<grid, 128 * g, smem, st>>>(S, K, desc, ct_a, ct_b, abar_in, max_steps, ext, acc_out, count);
    return cudaGetLastError();
}

void team_capacities(const LaunchShape &S, uint32_t cap[3]) {
    cap[0] = cap[1] = cap[2] = 0;
    if (!warp_form_supported(S) || !br::teams_fit_tmem()) return;
    cap[0] = br::team_capacity<1>(S.k, S.n);
    cap[1] = br::team_capacity<2>(S.k, S.n);
    cap[2] = br::team_capacity<3>(S.k, S.n);
}

namespace {
// Clocks of an SM (in thousands) that a CMux step takes, measured on GB300:
// a full wave of the team kernel with 1, 2 and 3 teams a CTA (the same for k =
// 1 to 8, polynomials run side by side; one share buffer costs a second
// cluster barrier), and a pass of the warp kernel with 1, 2 and 3 gates a CTA,
// per transform slot (k + 2 slots a step).
constexpr double kTeamStep[3] = {14.2, 15.7, 19.5}, kOneBuffer = 2.5, kWarpSlot[3] = {6.8, 9.4, 11.0};
// A pass of the shared kernel (a gate per SM), k = 2 to 8.
constexpr double kSharedStep[7] = {19.2, 21.3, 27.2, 29.3, 31.9, 38.1, 40.2};

double team_cost(const LaunchShape &S, uint32_t count, int t) {
    if (!S.team_cap[t]) return 1e30;
    const double step = kTeamStep[t] + (br::team_layout(S.k, S.n, t + 1).share_buffers == 1 ? kOneBuffer : 0.0);
    return step * ((count + S.team_cap[t] - 1) / S.team_cap[t]);
}

double warp_cost(const LaunchShape &S, uint32_t count, uint32_t sms) {
    const uint32_t g = warp_gates(S.k, S.n, 0xFFFFFFFFu / 2, sms), pass = g * sms;
    if (g == 0) return 1e30;
    const uint32_t rest = count % pass;
    return (S.k + 2) * ((count / pass) * kWarpSlot[g - 1] + (rest ? kWarpSlot[(rest - 1) / sms] : 0.0));
}

bool shared_form_supported(const LaunchShape &S) {
    return warp_form_supported(S) && S.k >= 2 && br::shared_layout(S.k, S.n).total <= kWarpSmemMax;
}

// The shared kernel is the default variant's: it runs batches that the batched variants would.
double shared_cost(const LaunchShape &S, uint32_t count, uint32_t sms) {
    if (S.variant != 2 || !shared_form_supported(S) || S.k > 8) return 1e30;
    return kSharedStep[S.k - 2] * ((count + sms - 1) / sms);
}

cudaError_t launch_bootstrap_shared(const LaunchShape &S, const DeviceKeys &K, const GateDesc *desc,
                                    const uint32_t *ct_a, const uint32_t *ct_b, const uint32_t *abar_in,
                                    int64_t max_steps, uint32_t *ext, uint32_t *acc_out, uint32_t count,
                                    cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const size_t smem = br::shared_layout(S.k, S.n).total;
    auto kern = br::bootstrap_shared_kernel;
    e = br::allow_smem(kern);
    if (e != cudaSuccess) return e;
    const uint32_t grid = count < (uint32_t)sms ? count : (uint32_t)sms;
    kern<<<grid, 384, smem, st>>>(S, K, desc, ct_a, ct_b, abar_in, max_steps, ext, acc_out, count);
    return cudaGetLastError();
}

// The fastest kernel for this launch: the team kernel's teams a CTA, less one; 3: the shared kernel; -1: the warp
// kernel.  For the variants other than 2, -1 stands for their own kernel at the warp kernel's price, which is lower
// (1.6 to 1.8 times at k = 2): the team kernel is never taken where their own is faster, and given up earlier than it
// would have to be.
int fastest(const LaunchShape &S, uint32_t count, uint32_t sms, double &cost) {
    int best = -1;
    cost = warp_cost(S, count, sms);
    for (int t = 0; t < 4; ++t) {
        const double c = t < 3 ? team_cost(S, count, t) : shared_cost(S, count, sms);
        if (c < cost) cost = c, best = t;
    }
    return best;
}

uint32_t sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return (uint32_t)sms;
}

// The kernel of this launch, as `fastest` numbers them.
int team_choice(const LaunchShape &S, uint32_t count) {
    if (S.cluster_mode == MK_CLUSTER_OFF || !warp_form_supported(S)) return -1;
    if (S.cluster_mode == MK_CLUSTER_ON) {
        int best = 0;
        for (int t = 1; t < 3; ++t)
            if (team_cost(S, count, t) < team_cost(S, count, best)) best = t;
        return S.team_cap[best] ? best : -1;
    }
    const uint32_t sms = sm_count();
    double cost;
    return sms ? fastest(S, count, sms, cost) : -1;
}
}  // namespace

// A launch whose last pass would leave much of the chip idle: how many of its
// gates to run first, whole passes of a gate per SM each, so that the rest can
// have the kernel that is fastest for so few (0: all in one launch).  Two
// launches in turn cost their sum; 4 % covers the second's start.  Measured
// (GB300, blind rotation), one launch -> two: k = 2, 200 gates 19.8 -> 18.7 ms, 457 39.0 -> 30.0; k = 4, 200 58.6 -> 49.9,
// 465 116 -> 84.7, 1001 184 -> 169.6; k = 8, 200 174 -> 155.
uint32_t bootstrap_head(const LaunchShape &S, uint32_t count) {
    if (S.cluster_mode != MK_CLUSTER_AUTO || S.variant != 2 || !warp_form_supported(S) || S.k > 8 ||
        !(S.team_cap[0] | S.team_cap[1] | S.team_cap[2]))
        return 0;
    const uint32_t sms = sm_count();
    if (sms == 0 || count <= sms) return 0;
    double whole, first, rest;
    fastest(S, count, sms, whole);
    double best = 0.96 * whole;
    uint32_t head = 0;
    for (uint32_t h = sms; h < count; h += sms) {
        fastest(S, h, sms, first);
        fastest(S, count - h, sms, rest);
        if (first + rest < best) best = first + rest, head = h;
    }
    return head;
}

bool team_form_chosen(const LaunchShape &S, uint32_t count) { return team_choice(S, count) >= 0; }
bool shared_form_chosen(const LaunchShape &S, uint32_t count) { return team_choice(S, count) == 3; }

cudaError_t launch_bootstrap_team(const LaunchShape &S, const DeviceKeys &K, const GateDesc *desc,
                                  const uint32_t *ct_a, const uint32_t *ct_b, const uint32_t *abar_in,
                                  int64_t max_steps, uint32_t *ext, uint32_t *acc_out, uint32_t count,
                                  cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    if (K.tw_warp == nullptr || K.status == nullptr) return cudaErrorInvalidValue;
    switch (team_choice(S, count)) {
        case 0: return br::launch_team<1>(S, K, desc, ct_a, ct_b, abar_in, max_steps, ext, acc_out, count, st);
        case 1: return br::launch_team<2>(S, K, desc, ct_a, ct_b, abar_in, max_steps, ext, acc_out, count, st);
        case 2: return br::launch_team<3>(S, K, desc, ct_a, ct_b, abar_in, max_steps, ext, acc_out, count, st);
        case 3: return launch_bootstrap_shared(S, K, desc, ct_a, ct_b, abar_in, max_steps, ext, acc_out, count, st);
        default: return cudaErrorInvalidConfiguration;
    }
}

bool small_form_supported(const LaunchShape &S) {
    return S.form == MK_FORM_NTT2 && S.logN == 8 && S.d == 3 && S.bg_bit == 8 && S.k <= 8 &&
           br::small_layout(S.k, S.n).total <= kWarpSmemMax;
}

cudaError_t launch_bootstrap_small(const LaunchShape &S, const DeviceKeys &K, const GateDesc *desc,
                                   const uint32_t *ct_a, const uint32_t *ct_b, const uint32_t *abar_in,
                                   int64_t max_steps, uint32_t *ext, uint32_t *acc_out, uint32_t count,
                                   cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    if (!small_form_supported(S) || K.tw_split == nullptr) return cudaErrorInvalidValue;
    const size_t smem = br::small_layout(S.k, S.n).total;
    auto run = [&](auto kern) {
        const cudaError_t e = br::allow_smem(kern);
        if (e != cudaSuccess) return e;
        kern<<<count, 64 * (S.k + 1), smem, st>>>(S, K, desc, ct_a, ct_b, abar_in, max_steps, ext, acc_out);
        return cudaGetLastError();
    };
    if (S.k > 3) return run(br::bootstrap_small_kernel<8, 1>);
    // one gate an SM: all the registers; more: three CTAs an SM (600 gates at k = 2 1.38 ms, with two 1.45)
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    return count <= (uint32_t)sms ? run(br::bootstrap_small_kernel<3, 1>) : run(br::bootstrap_small_kernel<3, 3>);
}
}  // namespace mk
