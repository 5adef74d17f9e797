// mk_bootstrap_team.cuh -- the latency form of the two-prime blind rotation at
// N = 1024, base 2^8: one gate per thread-block cluster, one team of four
// warps per accumulator polynomial.
//
// The warp kernel (mk_bootstrap_warp.cuh) gives a gate four warps that take
// the k + 1 polynomials of a CMux step one after the other: 27.8 k clocks a
// step at k = 2 when a gate has an SM to itself, most of them waits.  Here
// team jj owns ACC_jj and, per step (hybrid product as in mk_bootstrap.cuh),
//   1. cuts the digits of its (X^-e - 1) ACC_jj, transforms them (tcgen05 and
//      register stages of the warp kernel) and forms c'_jj = <u_jj, d> and its
//      share v_jj = <u_jj, A_jj>, which it stores into the CTAs that hold
//      polynomials 0 and i (distributed shared memory);
//   2. arrives at the cluster barrier; a team that owns neither 0 nor i
//      inverse-transforms c'_jj into ACC_jj before it waits there;
//   3. in each of those CTAs one team sums the shares, inverse-transforms v
//      and starts the products of its digits; the teams of 0 and i take the
//      result from TMEM, add <w, f0> or <w, f1> to their c' and
//      inverse-transform it into their ACC.
// One cluster barrier a step; v's transform is done twice when 0 and i are in
// different CTAs, which costs no time: those SMs would wait.
//
// T teams a CTA, ceil((k + 1) / T) CTAs a cluster.  T = 1 has the shortest
// step (a team has the SM's four schedulers to itself); T = 2 and 3 put more
// gates on the chip at once.  Measured (GB300, blind rotation of one wave):
// k = 2: 1 gate 6.4 ms (the cluster kernel it replaces 11.5, the warp kernel
// 15.7), 37 gates 7.7, 76 gates (T = 2) 8.4, 152 gates (T = 3) 10.7 against 14.3;
// k = 4: 1 gate 13.2 (23.7), 5 gates 13.5; k = 8: 1 gate 34.5 ms against 150.
// From about 77 gates the shared kernel (mk_bootstrap_shared.cuh) is faster.
// A step is a chain of dependent phases: at T = 1 about 11.8 k clocks, of them
// digits 0.6, two products 0.8 each, two sets of butterflies and key products
// 2.3 and 1.9, the cluster barrier 1.0, two inverse transforms 1.4 each.
// Waits for products are bounded (products_wait); a CTA whose wait ran out
// keeps passing the cluster barriers, so it strands no other (its results are
// garbage and mk_sync reports MK_ETIMEOUT).
#pragma once
#include <cooperative_groups.h>

#include "mk_bootstrap_warp.cuh"

namespace mk {
namespace br {

namespace cg = cooperative_groups;

// Shared memory of a CTA: tables, control block, per team accumulator, digits
// and transposition buffers, the shares of v (8 KB a polynomial; two buffers
// by step parity where they fit, else one and a second barrier a step), the
// mod-switched words.
struct TeamLayout {
    size_t ctl, team, team_bytes, shares, abar, total;
    size_t acc, digits, xbuf;
    uint32_t share_buffers;
};

__host__ __device__ inline TeamLayout team_layout(uint32_t k, uint32_t n, uint32_t teams) {
    TeamLayout L;
    L.ctl = (size_t)(teams == 3 ? Operands<3>::units : kTabSmall) * 16;
    L.team = L.ctl + ((sizeof(WarpCtl) + 15) & ~size_t(15));
    L.acc = 0;
    L.digits = 4096;
    L.xbuf = L.digits + 8 * kBUnit;
    L.team_bytes = L.xbuf + 8192;
    L.shares = L.team + L.team_bytes * teams;
    const size_t words = (sizeof(uint16_t) * (k * n + 1) + 15) & ~size_t(15), buffer = (size_t)8192 * (k + 1);
    L.share_buffers = L.shares + 2 * buffer + words <= kWarpSmemMax ? 2 : 1;
    L.abar = L.shares + L.share_buffers * buffer;
    L.total = L.abar + words;
    return L;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }

template <int T>
__global__ void __launch_bounds__(128 * T, 1)
bootstrap_team_kernel(LaunchShape S, DeviceKeys K, const GateDesc *__restrict__ desc,
                      const uint32_t *__restrict__ ct_a, const uint32_t *__restrict__ ct_b,
                      const uint32_t *__restrict__ abar_in, int64_t max_steps, uint32_t *__restrict__ ext,
                      uint32_t *__restrict__ acc_out) {
    constexpr int N = 1024;
    constexpr int POLY = N / 2;  // 16-byte units of a key polynomial (a plane of 256 per prime)
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int k = (int)S.k, n = (int)S.n, cta = (int)cluster.block_rank();
    const uint32_t ctas = (uint32_t)(k + T) / T, gate = blockIdx.x / ctas;
    const TeamLayout L = team_layout(S.k, S.n, T);
    uint4 *tab = reinterpret_cast<uint4 *>(smem);
    {
        const uint4 *src = static_cast<const uint4 *>(K.tw_warp);
        for (int u = threadIdx.x; u < Operands<T>::units; u += 128 * T) tab[u] = src[u];
    }
    WarpCtl *ctl = reinterpret_cast<WarpCtl *>(smem + L.ctl);
    constexpr uint32_t columns = Operands<T>::columns;
    if (threadIdx.x == 0) {
        for (int g = 0; g < kWarpMaxGates; ++g) st_mbar_init(st_smem_addr(&ctl->bar[g]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        ctl->abort = 0;
    }
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(st_smem_addr(&ctl->tmem)),
                     "r"(columns)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    uint16_t *abar = reinterpret_cast<uint16_t *>(smem + L.abar);
    if (abar_in) {
        const uint32_t W = S.k * S.n + 1;
        for (uint32_t x = threadIdx.x; x < W; x += 128 * T) abar[x] = (uint16_t)abar_in[(size_t)gate * W + x];
    } else {
        lin_modswitch(S, desc[gate], ct_a, ct_b, abar, threadIdx.x, 128 * T);
    }
    st_fence_proxy_async();  // the tables are operands of the matrix products
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const int wid = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);
    if (wid < 4) fill_operands<T>(ctl->tmem, static_cast<const uint4 *>(K.tw_warp), wid, threadIdx.x & 31);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const int lane = threadIdx.x & 31, warp = wid & 3, slot = wid >> 2, t128 = threadIdx.x & 127;
    const int pr = warp >> 1, h = warp & 1, bar = 1 + slot;
    const int jj = cta * T + slot;  // this team's polynomial
    const bool active = jj <= k;
    unsigned char *tm = smem + L.team + L.team_bytes * slot;
    uint32_t *acc = reinterpret_cast<uint32_t *>(tm + L.acc);
    uint4 *digits = reinterpret_cast<uint4 *>(tm + L.digits);
    uint32_t *ex = reinterpret_cast<uint32_t *>(tm + L.xbuf), *xb = ex + 512 * warp;
    uint4 *shares = reinterpret_cast<uint4 *>(smem + L.shares);
    const uint4 *heap = tab + warp * 256 + lane, *heap_rev = tab + (warp ^ 1) * 256 + 31 - lane;
    const uint4 *rows = tab + kTabHalves + pr * 16;
    const uint4 *crosses = tab + kTabHalves + kTabRows;
    const uint32_t ones_s = st_smem_addr(crosses + kTabCross), plane0_s = ones_s + 16 * kTabOnes;
    const uint32_t digits_s = st_smem_addr(digits);
    const uint32_t mbar0 = st_smem_addr(&ctl->bar[0]), tmem0 = ctl->tmem, lanes = (uint32_t)(32 * warp) << 16;
    const PrimeK q = prime_of(pr, S.d - 3);
    const Gadget gad = make_gadget(8);
    const uint4 *bk_all = static_cast<const uint4 *>(K.bk) + pr * (POLY / 2);
    const uint4 *key_a = static_cast<const uint4 *>(K.keyA) + (size_t)jj * 3 * POLY + pr * (POLY / 2);
    const int all_steps = k * n;
    const int limit = (max_steps >= 0 && max_steps < all_steps) ? (int)max_steps : all_steps;
    const uint32_t m0 = (lane & 15) + 32 * (2 * warp + (lane >> 4)), sw0 = acc_pos(m0);
    uint4 *unit = digits + (2 * warp + (lane >> 4)) * (kBUnit / 16) + (lane & 15);
    const uint32_t half_odd = 4 * (lane & 1), eighth = 16 * h + (lane >> 1);
    uint32_t phase[T];  // products completed by each team of this CTA
#pragma unroll
    for (int s = 0; s < T; ++s) phase[s] = 0;

    auto start_products = [&](bool issue) {
        st_fence_proxy_async();
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        quad_sync(bar);
        if (warp == 0 && issue && elect_one()) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            issue_products<T>(tmem0, tmem0 + 144 * slot, ones_s, plane0_s, digits_s, mbar0 + 8 * slot);
        }
        __syncwarp();
    };
    auto wait_products = [&](int s, uint32_t ph) {
        if (!st_mbar_try(mbar0 + 8 * s, ph & 1)) products_wait(mbar0 + 8 * s, ph & 1, &ctl->abort, S.wait_ns, K.status);
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    };
    auto load_products = [&](uint32_t(&x)[3][16], int s) {
        const uint32_t tmem = tmem0 + 144 * s + lanes;
        PlaneSums f[2];  // a digit's sums are on their way while the one before is combined
        fetch_sums(f[0], tmem);
        sums_fetched();
        fetch_sums(f[1], tmem + 16);
        combine_planes(x[0], f[0], q);
        sums_fetched();
        fetch_sums(f[0], tmem + 32);
        combine_planes(x[1], f[1], q);
        sums_fetched();
        combine_planes(x[2], f[0], q);
    };
    auto butterflies = [&](uint32_t(&x)[3][16]) {
        half_stage<3, 3>(x, heap, q);
        half_stage<3, 2>(x, heap, q);
        half_stage<3, 1>(x, heap, q);
        half_stage<3, 0>(x, heap, q);
    };

    if (active) {
        const uint32_t bbar = abar[k * n];
        for (uint32_t m = t128; m < (uint32_t)N; m += 128) {
            const uint32_t r = (m + bbar) & (2 * N - 1);
            acc[acc_pos(m)] = jj ? 0u : ((r >= (uint32_t)N) ? (0u - (1u << 29)) : (1u << 29));
        }
        quad_sync(bar);
    }
    cluster_arrive();  // every CTA of the cluster is running before remote stores
    cluster_wait();
    uint32_t parity = 0;
    int i = 1, left = n;  // party of the step, steps left of it
    uint32_t e_next = abar[0];
#pragma unroll 1
    for (int step = 0; step < limit; ++step) {
        const uint32_t e = e_next;
        e_next = abar[step + 1];  // (the last one reads b's word)
        if (left == 0) {
            left = n;
            ++i;
        }
        --left;
        if (e == 0) continue;  // the same word in every CTA: the whole cluster skips
        const int cta_i = i / T;
        // The team of this CTA that transforms v, if the CTA holds polynomial 0 or i
        const int vteam = cta == 0 ? 0 : (cta == cta_i ? i % T : -1);
        const bool last = jj == 0 || jj == i;
        const uint4 *bk = bk_all + (size_t)step * 9 * POLY;
        const bool issue = step != S.skip_key_step;
        uint32_t C[16];
        if (active) {
            // 1. c'_jj and v_jj
            {
                uint32_t w[8];
#pragma unroll
                for (int i8 = 0; i8 < 8; ++i8) {
                    const uint32_t r = m0 + 16 * (i8 & 1) + 256 * (i8 >> 1) + e;
                    const uint32_t a = acc[acc_pos(r & (N - 1))];
                    const uint32_t neg = (uint32_t)((int32_t)(r << 21) >> 31);  // bit 10 of r: -1
                    w[i8] = (a ^ neg) - neg - acc[(sw0 ^ (16 * (i8 & 1))) + 256 * (i8 >> 1)] + gad.offset;
                }
                store_digits(unit, w);
            }
            start_products(issue);
            constexpr int AHEAD = T == 1 ? 4 : 1;  // key groups on their way during the products and butterflies
            uint4 key[AHEAD][6];
#pragma unroll
            for (int v = 0; v < AHEAD; ++v) load_keys(key[v], bk, key_a, half_odd + v, eighth);
            uint32_t x[3][16];
            wait_products(slot, phase[slot]);
            load_products(x, slot);
            butterflies(x);
            uint32_t V[16];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
#pragma unroll
                for (int e4 = 0; e4 < 4; ++e4) {
                    const int c = 4 * v + e4;
                    const uint4(&kv)[6] = key[v % AHEAD];
                    C[c] = mac3_redc(x[0][c], x[1][c], x[2][c], word_of(kv[0], e4), word_of(kv[1], e4), word_of(kv[2], e4), q);
                    V[c] = mac3_redc(x[0][c], x[1][c], x[2][c], word_of(kv[3], e4), word_of(kv[4], e4), word_of(kv[5], e4), q);
                }
                if (v + AHEAD < 4) load_keys(key[v % AHEAD], bk, key_a, half_odd + v + AHEAD, eighth);
            }
            uint4 *mine = shares + (size_t)parity * 512 * (k + 1) + 512 * jj + t128;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (r == 1 && cta_i == 0) break;
                uint4 *dst = cluster.map_shared_rank(mine, r ? cta_i : 0);
#pragma unroll
                for (int v = 0; v < 4; ++v) dst[128 * v] = make_uint4(V[4 * v], V[4 * v + 1], V[4 * v + 2], V[4 * v + 3]);
            }
        }
#pragma unroll
        for (int s = 0; s < T; ++s) ++phase[s];
        __syncwarp();
        cluster_arrive();
        uint32_t z[8];
        if (active && !last) {
            // 2. this polynomial is done
            inverse_crt(C, z, heap_rev, rows, crosses + pr * 16, crosses, xb, ex, q, h, warp, lane, bar);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[(sw0 ^ (16 * (c & 1))) + 256 * (c >> 1)] += z[c];
            quad_sync(bar);
        }
        const uint4 *kf = bk + (jj == 0 ? 3 : 6) * POLY;
        constexpr int FAHEAD = T == 1 ? 4 : 1;
        uint4 key[FAHEAD][3];
        if (last) {
#pragma unroll
            for (int v = 0; v < FAHEAD; ++v) load_key(key[v], kf, half_odd + v, eighth);
        }
        __syncwarp();
        cluster_wait();  // every share of v has arrived
        if (last) {
            // 3. w = g^-1(v), c'_0 += <w, f0>, c'_i += <w, f1>
            if (slot == vteam) {
                uint32_t y[16];
                const uint4 *src = shares + (size_t)parity * 512 * (k + 1) + t128;
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const uint4 a = src[128 * v];
                    y[4 * v] = a.x, y[4 * v + 1] = a.y, y[4 * v + 2] = a.z, y[4 * v + 3] = a.w;
                }
                for (int s = 1; s <= k; ++s)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const uint4 a = src[512 * s + 128 * v];
#pragma unroll
                        for (int e4 = 0; e4 < 4; ++e4) {
                            const uint32_t t = y[4 * v + e4] + word_of(a, e4);  // each below 4 p
                            y[4 * v + e4] = min(t, t - q.p4);
                        }
                    }
                inverse_crt(y, z, heap_rev, rows, crosses + pr * 16, crosses, xb, ex, q, h, warp, lane, bar);
#pragma unroll
                for (int c = 0; c < 8; ++c) z[c] += gad.offset;
                store_digits(unit, z);
                start_products(issue);
            }
            uint32_t x[3][16];
            // both teams of a CTA that holds 0 and i read the same products
            wait_products(vteam, phase[vteam]);
            load_products(x, vteam);
            if (T > 1 && cta == 0 && cta_i == 0) {  // before the transforming team reuses its columns
                asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                asm volatile("bar.sync 8, 256;\n" ::: "memory");
            }
            butterflies(x);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
#pragma unroll
                for (int e4 = 0; e4 < 4; ++e4) {
                    const int c = 4 * v + e4;
                    const uint4(&kv)[3] = key[v % FAHEAD];
                    const uint32_t a = C[c] + mac3_redc(x[0][c], x[1][c], x[2][c], word_of(kv[0], e4), word_of(kv[1], e4),
                                                        word_of(kv[2], e4), q);
                    C[c] = min(a, a - q.p4);
                }
                if (v + FAHEAD < 4) load_key(key[v % FAHEAD], kf, half_odd + v + FAHEAD, eighth);
            }
            inverse_crt(C, z, heap_rev, rows, crosses + pr * 16, crosses, xb, ex, q, h, warp, lane, bar);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[(sw0 ^ (16 * (c & 1))) + 256 * (c >> 1)] += z[c];
            quad_sync(bar);
        }
#pragma unroll
        for (int s = 0; s < T; ++s)
            if (s == vteam) ++phase[s];
        if (L.share_buffers == 2) {
            parity ^= 1;
        } else {  // one buffer: every share is read before the next step's are stored
            __syncwarp();
            cluster_arrive();
            cluster_wait();
        }
    }
    if (active) {
        if (acc_out) {
            uint32_t *dst = acc_out + ((size_t)gate * (k + 1) + jj) * N;
            for (uint32_t x = t128; x < (uint32_t)N; x += 128) dst[x] = acc[acc_pos(x)];
        } else {
            uint32_t *dst = ext + (size_t)gate * (k * N + 1);
            if (jj == 0) {
                if (t128 == 0) dst[k * N] = acc[0] + (1u << 29);  // +1/8
            } else {
                for (int m = t128; m < N; m += 128) dst[(jj - 1) * N + m] = m == 0 ? acc[0] : 0u - acc[acc_pos(N - m)];
            }
        }
    }
    release_tmem<columns, (size_t)Operands<T>::units * 16 + offsetof(WarpCtl, tmem), true>(K.status);
    cluster_arrive();  // no CTA leaves while another could still store into its shared memory
    cluster_wait();
}

template <int T>
cudaLaunchConfig_t team_config(uint32_t k, uint32_t n, uint32_t count, cudaStream_t st, cudaLaunchAttribute *attr) {
    const uint32_t ctas = (k + T) / T;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(count * ctas, 1, 1);
    cfg.blockDim = dim3(128 * T, 1, 1);
    cfg.dynamicSmemBytes = team_layout(k, n, T).total;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Registers that a CTA takes from its SM (allocated in units of 8 a thread).
template <int T>
uint32_t team_registers() {
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, bootstrap_team_kernel<T>) != cudaSuccess) return 0;
    return (uint32_t)((a.numRegs + 7) / 8 * 8) * 128 * T;
}

// Whether no SM can hold CTAs of these kernels that want more than its 512
// TMEM columns together, from one launch or from several streams'.  An
// allocation waits until columns are free, and a CTA that has its own waits
// for its cluster: two clusters, each holding an SM's columns that the other
// asks for, would wait for ever, and occupancy queries know nothing of TMEM.
// T = 1 (256 columns) may have two CTAs an SM, T = 2 and 3 (512) must be alone
// among them.  Registers see to it (255, 236 and 168 a thread of 65536); they
// are the compiler's choice, so they are checked.  (Kernels without clusters
// only delay each other: whoever holds columns gets to its end.)
inline bool teams_fit_tmem() {
    static_assert(Operands<1>::columns == 256 && Operands<2>::columns == 512 && Operands<3>::columns == 512, "TMEM columns");
    int dev = 0, file = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&file, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess)
        return false;
    const uint32_t r1 = team_registers<1>(), r2 = team_registers<2>(), r3 = team_registers<3>(), all = (uint32_t)file;
    const uint32_t least = r1 < r2 ? (r1 < r3 ? r1 : r3) : (r2 < r3 ? r2 : r3);
    return 3 * r1 > all && r2 + least > all && r3 + least > all;
}

// Gates of this shape that can be resident at once, or 0 if none can.
template <int T>
uint32_t team_capacity(uint32_t k, uint32_t n) {
    const size_t smem = team_layout(k, n, T).total;
    if ((k + T) / T > 8 || smem > kWarpSmemMax) return 0;
    auto kern = bootstrap_team_kernel<T>;
    if (allow_smem(kern) != cudaSuccess) return 0;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = team_config<T>(k, n, 1, nullptr, attr);
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess) return 0;
    return (uint32_t)clusters;
}

template <int T>
cudaError_t launch_team(const LaunchShape &S, const DeviceKeys &K, const GateDesc *desc, const uint32_t *ct_a,
                        const uint32_t *ct_b, const uint32_t *abar_in, int64_t max_steps, uint32_t *ext,
                        uint32_t *acc_out, uint32_t count, cudaStream_t st) {
    auto kern = bootstrap_team_kernel<T>;
    const cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = team_config<T>(S.k, S.n, count, st, attr);
    return cudaLaunchKernelEx(&cfg, kern, S, K, desc, ct_a, ct_b, abar_in, max_steps, ext, acc_out);
}

}  // namespace br
}  // namespace mk
