// mk_bootstrap_shared.cuh -- the two-prime blind rotation at N = 1024, base
// 2^8, d = 3, k >= 2: one gate per CTA, the accumulator polynomials shared out
// among three teams of four warps.
//
// Up to one gate per SM the warp kernel (mk_bootstrap_warp.cuh) has four warps
// on an SM, one for each scheduler: a transform slot takes 6.8 k clocks where
// three gates' slots side by side take 11.0 k.  The team kernel needs k + 1
// teams a gate, so many parties put few gates on the chip.  Here the same
// three teams that fill an SM work on one gate.  Per CMux step of party i
// (hybrid product as in mk_bootstrap.cuh):
//   A. team 0 takes some of the other parties' polynomials, then 0; team 1
//      some of the others, then i; team 2 the rest.  For each: digits of
//      (X^-e - 1) ACC_jj, their products and butterflies (a polynomial's
//      products run under the one before), c'_jj = <u_jj, d> and v += <u_jj,
//      A_jj>.  Another party's c'_jj is inverse-transformed into its ACC at
//      once; c'_0 and c'_i stay in registers;
//   B. teams 1 and 2 hand their shares of v to team 0, which inverse-transforms
//      v and starts the products of its digits; teams 0 and 1 both read them
//      from TMEM and finish ACC_0 and ACC_i.
// Team 2 has no part in B and goes on with the next step, so it takes the
// larger share of A (others_of).
//
// Measured (GB300, blind rotation, one gate per SM, against the best of the
// team and warp kernels): 152 gates at k = 3 27.6 -> 17.3 ms, k = 4 39 -> 29.4,
// k = 5 60 -> 39.6, k = 6 86 -> 51.8, k = 7 113 -> 72; 96 gates at k = 8 134 -> 87 ms.
// At k = 6 a step takes 31.9 k clocks of an SM against the 29.3 k of the warp
// kernel's rate with three gates side by side: the multiply pipe bounds it, and
// for few parties the chain of phase B does.
//
// Hand-over, by named barriers (at 4 and 7 the one who gives does not wait):
//   4: teams 1 and 2 have stored their shares; team 0 waits.
//   7: team 0 has read them; team 2 waits before it stores the next step's.
//   6: teams 0 and 1 have read v's products; both wait, so team 1 is never a
//      step ahead of team 0 whatever became of a wait for products: without
//      that it would arrive at 4 twice after a wait that ran out.
// v's products have an mbarrier of their own, one phase a step.
// Where the party changes the polynomials change hands: all teams meet (9).
// Waits for products are bounded (products_wait) and nothing branches on their
// outcome, so no team misses a barrier.
#pragma once
#include "mk_bootstrap_team.cuh"

namespace mk {
namespace br {

struct SharedCtl {
    unsigned long long bar[4];  // mbarriers: the teams' products, v's
    uint32_t tmem, abort;
};
struct SharedLayout {
    size_t ctl, acc, team, team_bytes, shares, abar, total;
    size_t digits, xbuf;
};
__host__ __device__ inline SharedLayout shared_layout(uint32_t k, uint32_t n) {
    SharedLayout L;
    L.ctl = (size_t)Operands<3>::units * 16;
    L.acc = L.ctl + ((sizeof(SharedCtl) + 15) & ~size_t(15));
    L.team = L.acc + (size_t)4096 * (k + 1);
    L.digits = 0;
    L.xbuf = 8 * kBUnit;
    L.team_bytes = L.xbuf + 8192;
    L.shares = L.team + 3 * L.team_bytes;
    L.abar = L.shares + 2 * 8192;
    L.total = L.abar + ((sizeof(uint16_t) * (k * n + 1) + 15) & ~size_t(15));
    return L;
}

// Of the k - 1 other parties' polynomials, how many each team takes.  Phase B
// keeps teams 0 and 1 busy for about as long as 1.5 slots of phase A; team 2
// with (k + 2) / 3 or (k + 4) / 3 of them measured 0 to 22 % slower (152 gates,
// k = 3 to 8), team 1 with the odd one 3 % at k = 4.
struct Others {
    int first[3], count[3];
};
__host__ __device__ inline Others others_of(int k) {
    Others o;
    const int m = k - 1, two = (k + 3) / 3;
    o.count[2] = two < m ? two : m;
    o.count[0] = (m - o.count[2] + 1) / 2;
    o.count[1] = m - o.count[2] - o.count[0];
    o.first[0] = 0;
    o.first[1] = o.count[0];
    o.first[2] = o.count[0] + o.count[1];
    return o;
}

__global__ void __launch_bounds__(384, 1)
bootstrap_shared_kernel(LaunchShape S, DeviceKeys K, const GateDesc *__restrict__ desc,
                        const uint32_t *__restrict__ ct_a, const uint32_t *__restrict__ ct_b,
                        const uint32_t *__restrict__ abar_in, int64_t max_steps, uint32_t *__restrict__ ext,
                        uint32_t *__restrict__ acc_out, uint32_t count) {
    constexpr int N = 1024;
    constexpr int POLY = N / 2;  // 16-byte units of a key polynomial (a plane of 256 per prime)
    extern __shared__ __align__(16) unsigned char smem[];
    const int k = (int)S.k, n = (int)S.n;
    const SharedLayout L = shared_layout(S.k, S.n);
    uint4 *tab = reinterpret_cast<uint4 *>(smem);
    {
        const uint4 *src = static_cast<const uint4 *>(K.tw_warp);
        for (int u = threadIdx.x; u < Operands<3>::units; u += 384) tab[u] = src[u];
    }
    SharedCtl *ctl = reinterpret_cast<SharedCtl *>(smem + L.ctl);
    constexpr uint32_t columns = Operands<3>::columns;
    if (threadIdx.x == 0) {
        for (int g = 0; g < 4; ++g) st_mbar_init(st_smem_addr(&ctl->bar[g]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        ctl->abort = 0;
    }
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(st_smem_addr(&ctl->tmem)),
                     "r"(columns)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    st_fence_proxy_async();  // the tables are operands of the matrix products
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const int wid = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);
    if (wid < 4) fill_operands<3>(ctl->tmem, static_cast<const uint4 *>(K.tw_warp), wid, threadIdx.x & 31);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const int lane = threadIdx.x & 31, warp = wid & 3, team = wid >> 2, t128 = threadIdx.x & 127;
    const int pr = warp >> 1, h = warp & 1, bar = 1 + team;
    uint32_t *acc = reinterpret_cast<uint32_t *>(smem + L.acc);
    unsigned char *tm = smem + L.team + L.team_bytes * team;
    uint4 *digits = reinterpret_cast<uint4 *>(tm + L.digits);
    uint32_t *ex = reinterpret_cast<uint32_t *>(tm + L.xbuf), *xb = ex + 512 * warp;
    uint4 *shares = reinterpret_cast<uint4 *>(smem + L.shares);
    uint16_t *abar = reinterpret_cast<uint16_t *>(smem + L.abar);
    const uint4 *heap = tab + warp * 256 + lane, *heap_rev = tab + (warp ^ 1) * 256 + 31 - lane;
    const uint4 *rows = tab + kTabHalves + pr * 16;
    const uint4 *crosses = tab + kTabHalves + kTabRows;
    const uint32_t ones_s = st_smem_addr(crosses + kTabCross), plane0_s = ones_s + 16 * kTabOnes;
    const uint32_t digits_s = st_smem_addr(digits);
    const uint32_t mbar = st_smem_addr(&ctl->bar[team]), vbar = st_smem_addr(&ctl->bar[3]);
    const uint32_t tmem0 = ctl->tmem, tmem = tmem0 + 144 * team, lanes = (uint32_t)(32 * warp) << 16;
    const PrimeK q = prime_of(pr, S.d - 3);
    const Gadget gad = make_gadget(8);
    const uint4 *bk_all = static_cast<const uint4 *>(K.bk) + pr * (POLY / 2);
    const uint4 *keyA = static_cast<const uint4 *>(K.keyA) + pr * (POLY / 2);
    const int all_steps = k * n;
    const int limit = (max_steps >= 0 && max_steps < all_steps) ? (int)max_steps : all_steps;
    const uint32_t m0 = (lane & 15) + 32 * (2 * warp + (lane >> 4)), sw0 = acc_pos(m0);
    uint4 *unit = digits + (2 * warp + (lane >> 4)) * (kBUnit / 16) + (lane & 15);
    const uint32_t half_odd = 4 * (lane & 1), eighth = 16 * h + (lane >> 1);
    const Others others = others_of(k);
    const int mine = others.count[team], first = others.first[team];
    const int slots = mine + (team < 2 ? 1 : 0);  // phase A; teams 0 and 1 have one more, v's
    uint32_t phase = 0, vphase = 0;               // products waited for
    bool reading = false;                         // team 2: a step's shares may still be being read

    // The digits of (X^-e - 1) ACC_jj, and the issue of their products by an elected lane (lane 0: 152 gates at
    // k = 4 31.4 against 30.1 ms).
    auto cut_digits = [&](int jj, uint32_t e) {
        const uint32_t *ap = acc + jj * N;
        uint32_t w[8];
#pragma unroll
        for (int i8 = 0; i8 < 8; ++i8) {
            const uint32_t r = m0 + 16 * (i8 & 1) + 256 * (i8 >> 1) + e;
            const uint32_t a = ap[acc_pos(r & (N - 1))];
            const uint32_t neg = (uint32_t)((int32_t)(r << 21) >> 31);  // bit 10 of r: -1
            w[i8] = (a ^ neg) - neg - ap[(sw0 ^ (16 * (i8 & 1))) + 256 * (i8 >> 1)] + gad.offset;
        }
        store_digits(unit, w);
    };
    auto start_products = [&](uint32_t to, bool issue) {
        st_fence_proxy_async();
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        quad_sync(bar);
        if (warp == 0 && issue && elect_one()) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            issue_products<3>(tmem0, tmem, ones_s, plane0_s, digits_s, to);
        }
        __syncwarp();
    };
    auto next_step = [&](int s) {  // e = 0: X^0 - 1 = 0, every digit is 0, the product adds nothing
        while (s < limit && abar[s] == 0) ++s;
        return s;
    };

    for (uint32_t gate = blockIdx.x; gate < count; gate += gridDim.x) {
        if (abar_in) {
            const uint32_t W = S.k * S.n + 1;
            for (uint32_t x = threadIdx.x; x < W; x += 384) abar[x] = (uint16_t)abar_in[(size_t)gate * W + x];
        } else {
            lin_modswitch(S, desc[gate], ct_a, ct_b, abar, threadIdx.x, 384);
        }
        __syncthreads();
        {
            const uint32_t bbar = abar[k * n];
            for (uint32_t m = threadIdx.x; m < (uint32_t)N; m += 384) {
                const uint32_t r = (m + bbar) & (2 * N - 1);
                acc[acc_pos(m)] = (r >= (uint32_t)N) ? (0u - (1u << 29)) : (1u << 29);
            }
            for (uint32_t x = N + threadIdx.x; x < (uint32_t)(k + 1) * N; x += 384) acc[x] = 0;
        }
        __syncthreads();
        bool started = false;  // this step's first products are under way
        int next = 0, party = 1;
#pragma unroll 1
        for (int step = next_step(0); step < limit; step = next) {
            const int i = step / n + 1;
            const uint32_t e = abar[step];
            next = next_step(step + 1);
            const bool issue = step != S.skip_key_step;
            const uint4 *bk = bk_all + (size_t)step * 9 * POLY;
            if (i != party) {  // polynomials change hands
                asm volatile("bar.sync 9, 384;\n" ::: "memory");
                party = i;
            }
            // This team's polynomial in slot s: another party's, or at the end 0 or i
            auto poly_of = [&](int s) {
                if (s == mine) return team ? i : 0;
                const int o = first + s + 1;
                return o < i ? o : o + 1;
            };
            uint32_t V[16], C[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) V[c] = C[c] = 0;
            if (!started) {
                cut_digits(poly_of(0), e);
                start_products(mbar, issue);
            }
            // The next step's first products can start under this step's last slot if their polynomial is final
            // by then (team 0's once v's have left its columns).
            started = slots > 1 && next < limit && next / n + 1 == i;
            const int passes = slots + (team < 2 ? 1 : 0);
#pragma unroll 1
            for (int s = 0; s < passes; ++s) {
                const bool last = s == slots;  // v's products
                const uint32_t wb = last ? vbar : mbar, wp = last ? vphase : phase;
                if (!st_mbar_try(wb, wp & 1)) products_wait(wb, wp & 1, &ctl->abort, S.wait_ns, K.status);
                if (last)
                    ++vphase;
                else
                    ++phase;
                __syncwarp();
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                uint32_t x[3][16];
                {
                    const uint32_t from = (last ? tmem0 : tmem) + lanes;
                    load_factor(x[0], from, q);
                    load_factor(x[1], from + 16, q);
                    load_factor(x[2], from + 32, q);
                }
                if (last) {
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    asm volatile("bar.sync 6, 256;\n" ::: "memory");
                }
                // the next slot's products run under this one's butterflies
                const bool same = s + 1 < slots;
                if (same || (started && last == (team == 0))) {
                    cut_digits(poly_of(same ? s + 1 : 0), same ? e : abar[next]);
                    start_products(mbar, same ? issue : next != S.skip_key_step);
                }
                const int jj = last ? (team ? i : 0) : poly_of(s);
                const uint4 *k1 = bk + (last ? (team ? 6 : 3) * POLY : 0), *k2 = keyA + (size_t)jj * 3 * POLY;
                uint4 key[6];  // the first group is on its way during the butterflies
                if (last) {
                    load_key(reinterpret_cast<uint4(&)[3]>(key), k1, half_odd, eighth);
                } else {
                    load_keys(key, k1, k2, half_odd, eighth);
                }
                half_stage<3, 3>(x, heap, q);
                half_stage<3, 2>(x, heap, q);
                half_stage<3, 1>(x, heap, q);
                half_stage<3, 0>(x, heap, q);
                if (last) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
#pragma unroll
                        for (int e4 = 0; e4 < 4; ++e4) {
                            const int c = 4 * v + e4;
                            const uint32_t a = C[c] + mac3_redc(x[0][c], x[1][c], x[2][c], word_of(key[0], e4),
                                                                word_of(key[1], e4), word_of(key[2], e4), q);
                            C[c] = min(a, a - q.p4);
                        }
                        if (v < 3) load_key(reinterpret_cast<uint4(&)[3]>(key), k1, half_odd + v + 1, eighth);
                    }
                } else {
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
#pragma unroll
                        for (int e4 = 0; e4 < 4; ++e4) {
                            const int c = 4 * v + e4;
                            C[c] = mac3_redc(x[0][c], x[1][c], x[2][c], word_of(key[0], e4), word_of(key[1], e4),
                                             word_of(key[2], e4), q);
                            const uint32_t a = V[c] + mac3_redc(x[0][c], x[1][c], x[2][c], word_of(key[3], e4),
                                                                word_of(key[4], e4), word_of(key[5], e4), q);
                            V[c] = min(a, a - q.p4);
                        }
                        if (v < 3) load_keys(key, k1, k2, half_odd + v + 1, eighth);
                    }
                }
                const bool end_a = s == slots - 1;
                if (end_a && team) {  // this team's share of v
                    if (team == 2 && reading) asm volatile("bar.sync 7, 256;\n" ::: "memory");
                    uint4 *dst = shares + 512 * (team - 1) + t128;
#pragma unroll
                    for (int v = 0; v < 4; ++v) dst[128 * v] = make_uint4(V[4 * v], V[4 * v + 1], V[4 * v + 2], V[4 * v + 3]);
                    __threadfence_block();
                    asm volatile("bar.arrive 4, 384;\n" ::: "memory");
                    reading = true;
                    if (team == 1) continue;
                }
                uint32_t y[16], z[8];
                const bool sum = end_a && team == 0;
                if (sum) {
                    asm volatile("bar.sync 4, 384;\n" ::: "memory");
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const uint4 a = shares[128 * v + t128], b = shares[512 + 128 * v + t128];
#pragma unroll
                        for (int e4 = 0; e4 < 4; ++e4) {
                            uint32_t t = V[4 * v + e4] + word_of(a, e4);  // each below 4 p
                            t = min(t, t - q.p4) + word_of(b, e4);
                            y[4 * v + e4] = min(t, t - q.p4);
                        }
                    }
                    __threadfence_block();
                    asm volatile("bar.arrive 7, 256;\n" ::: "memory");
                } else {
#pragma unroll
                    for (int c = 0; c < 16; ++c) y[c] = C[c];
                }
                inverse_crt(y, z, heap_rev, rows, crosses + pr * 16, crosses, xb, ex, q, h, warp, lane, bar);
                if (sum) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) z[c] += gad.offset;
                    store_digits(unit, z);
                    start_products(vbar, issue);
                } else {
                    uint32_t *ap = acc + jj * N;
#pragma unroll
                    for (int c = 0; c < 8; ++c) ap[(sw0 ^ (16 * (c & 1))) + 256 * (c >> 1)] += z[c];
                    quad_sync(bar);
                }
            }
        }
        if (team == 2 && reading) {
            asm volatile("bar.sync 7, 256;\n" ::: "memory");
            reading = false;
        }
        __syncthreads();
        if (acc_out) {
            uint32_t *dst = acc_out + (size_t)gate * (k + 1) * N;
            for (uint32_t x = threadIdx.x; x < (uint32_t)(k + 1) * N; x += 384)
                dst[x] = acc[(x & ~(uint32_t)(N - 1)) + acc_pos(x & (N - 1))];
        } else {
            uint32_t *dst = ext + (size_t)gate * (k * N + 1);
            for (int i = 1; i <= k; ++i)
                for (int m = threadIdx.x; m < N; m += 384)
                    dst[(i - 1) * N + m] = m == 0 ? acc[i * N] : 0u - acc[i * N + acc_pos(N - m)];
            if (threadIdx.x == 0) dst[k * N] = acc[0] + (1u << 29);  // +1/8
        }
        __syncthreads();
    }
    release_tmem<columns, (size_t)Operands<3>::units * 16 + offsetof(SharedCtl, tmem), true>(K.status);
}

}  // namespace br
}  // namespace mk
