// mk_bootstrap_small.cuh -- the two-prime blind rotation at N = 256 (base 2^8,
// d = 3): one CTA per gate, one warp per (accumulator polynomial, prime).
//
// At N = 256 a transform is 32 lanes x 8 elements, so a warp holds one and
// needs no barrier inside it: three register passes with two exchanges
// through the warp's own shared memory.  The cluster kernel spent 12 k clocks a
// CMux step here (k = 2), nearly all of them on cluster and CTA barriers
// around a few hundred clocks of work.  Per step (hybrid product as in
// mk_bootstrap.cuh):
//   1. warp (jj, p) cuts the digits of its (X^-e - 1) ACC_jj, transforms the
//      three digit polynomials mod p, forms c'_jj and its share of v, and
//      stores the share;
//   2. one CTA barrier (shares double-buffered by step parity);
//   3. the pairs of 0 and i each sum the shares, inverse-transform v, cut and
//      transform its digits, add <w, f0> or <w, f1>; every pair inverse-
//      transforms its c' into its ACC.  The two warps of a pair meet at 64-thread
//      barriers to swap half of their residues for the recombination (CRT).
// Measured (GB300, blind rotation, toy set): k = 2, 1 to 24 gates 0.76 -> 0.50 ms
// (the cluster kernel), 600 gates 2.03 -> 1.38, 4000 gates 9.3 -> 9.1 (the batched
// kernel); k = 3, 600 gates 3.8 -> 2.5.
// Public keys stay in registers; a step's key words are loaded before its
// transforms.  Bounds as in mk_bootstrap_warp.cuh (lazy sums below 16 p).
#pragma once
#include "mk_bootstrap_warp.cuh"

namespace mk {
namespace br {

constexpr int kSmallN = 256;
// exchange position of index j: conflict-free for all layouts used here
__host__ __device__ constexpr int sx(int j) { return j + 4 * (j >> 5); }
constexpr int kSmallX = 288;  // words of an exchanged polynomial

struct SmallLayout {
    size_t tw, acc, xbuf, shares, vbuf, abar, total;
};
__host__ __device__ inline SmallLayout small_layout(uint32_t k, uint32_t n) {
    SmallLayout L;
    L.tw = 0;                                               // [2 directions][2 primes][N] {w, w'}
    L.acc = L.tw + 4 * kSmallN * 8;                         // [k + 1][N]
    L.xbuf = L.acc + (size_t)(k + 1) * kSmallN * 4;         // per warp three polynomials
    L.shares = L.xbuf + (size_t)2 * (k + 1) * 3 * kSmallX * 4;  // [2 parities][k + 1][2 primes][N]
    L.vbuf = L.shares + (size_t)2 * (k + 1) * 2 * kSmallN * 4;  // per pair
    L.abar = L.vbuf + (size_t)(k + 1) * kSmallN * 4;
    L.total = L.abar + ((sizeof(uint16_t) * (k * n + 1) + 15) & ~size_t(15));
    return L;
}

// Index of element c in the layout whose element bits are [LO, LO + 3).
template <int LO>
__device__ __forceinline__ int small_base(int lane) { return (lane & ((1 << LO) - 1)) | ((lane >> LO) << (LO + 3)); }

template <int NP, int FROM, int TO>
__device__ __forceinline__ void small_exchange(uint32_t (&x)[NP][8], uint32_t *buf, int lane) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        if constexpr (FROM == 0) {
            uint4 *dst = reinterpret_cast<uint4 *>(buf + p * kSmallX + sx(8 * lane));
            dst[0] = make_uint4(x[p][0], x[p][1], x[p][2], x[p][3]);
            dst[1] = make_uint4(x[p][4], x[p][5], x[p][6], x[p][7]);
        } else {
            const int b = small_base<FROM>(lane);
#pragma unroll
            for (int c = 0; c < 8; ++c) buf[p * kSmallX + sx(b | (c << FROM))] = x[p][c];
        }
    }
    __syncwarp();
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        if constexpr (TO == 0) {
            const uint4 *src = reinterpret_cast<const uint4 *>(buf + p * kSmallX + sx(8 * lane));
            const uint4 a = src[0], b = src[1];
            x[p][0] = a.x, x[p][1] = a.y, x[p][2] = a.z, x[p][3] = a.w;
            x[p][4] = b.x, x[p][5] = b.y, x[p][6] = b.z, x[p][7] = b.w;
        } else {
            const int b = small_base<TO>(lane);
#pragma unroll
            for (int c = 0; c < 8; ++c) x[p][c] = buf[p * kSmallX + sx(b | (c << TO))];
        }
    }
    __syncwarp();
}

// Forward stage at index bit B in layout LO.
template <int NP, int LO, int B>
__device__ __forceinline__ void small_fwd(uint32_t (&x)[NP][8], const uint2 *tw, int lane, const PrimeK &q) {
    constexpr int D = 1 << (B - LO);
    const int base = (1 << (7 - B)) + (small_base<LO>(lane) >> (B + 1));
#pragma unroll
    for (int g = 0; g < 4 / D; ++g) {
        const uint2 S = tw[base + g];
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int p = 0; p < NP; ++p) fwd_bf(x[p][2 * D * g + a], x[p][2 * D * g + a + D], S.x, S.y, q);
    }
}

// natural order (lane + 32 c), below 1.1 p -> bit-reversed order (8 lane + c), below 12 p
template <int NP>
__device__ __forceinline__ void small_forward(uint32_t (&x)[NP][8], const uint2 *tw, uint32_t *buf, int lane,
                                              const PrimeK &q) {
    small_fwd<NP, 5, 7>(x, tw, lane, q);
    small_fwd<NP, 5, 6>(x, tw, lane, q);
    small_fwd<NP, 5, 5>(x, tw, lane, q);
    small_exchange<NP, 5, 2>(x, buf, lane);
    small_fwd<NP, 2, 4>(x, tw, lane, q);
    small_fwd<NP, 2, 3>(x, tw, lane, q);
    small_fwd<NP, 2, 2>(x, tw, lane, q);
    small_exchange<NP, 2, 0>(x, buf, lane);
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int c = 0; c < 8; ++c) x[p][c] = min(x[p][c], x[p][c] - q.p8);  // below 13.1 p -> below 8 p
    small_fwd<NP, 0, 1>(x, tw, lane, q);
    small_fwd<NP, 0, 0>(x, tw, lane, q);
}

// Inverse stage at index bit B in layout LO; off(c): the bound of element c.
template <int LO, int B, class OFF>
__device__ __forceinline__ void small_inv(uint32_t (&y)[8], const uint2 *tw, int lane, const PrimeK &q, OFF off) {
    constexpr int D = 1 << (B - LO);
    const int base = (1 << (7 - B)) + (small_base<LO>(lane) >> (B + 1));
#pragma unroll
    for (int g = 0; g < 4 / D; ++g) {
        const uint2 S = tw[base + g];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const int c = 2 * D * g + a;
            const uint32_t u = y[c], v = y[c + D];
            y[c] = u + v;
            y[c + D] = shoup_k(u - v + off(c), S.x, S.y, q.p);
        }
    }
}

// bit-reversed order, below 4 p -> natural order, below 4 p
__device__ __forceinline__ void small_inverse(uint32_t (&x)[1][8], const uint2 *tw, uint32_t *buf, int lane,
                                              const PrimeK &q) {
    uint32_t(&y)[8] = x[0];
    // A pass of three stages on elements below 4 p: sums double the bound (8 p, 16 p), so the two elements at 16 p
    // are reduced before the third; products are below 2 p.
    auto off4 = [&](int) { return q.p4; };
    auto off_b = [&](int c) { return (c & 1) ? q.p2 : q.p8; };               // second stage: 2 p after a product, else 8 p
    auto off_c = [&](int c) { return (c & 3) == 1 ? q.p4 : q.p2; };           // third: 2 p (reduced), 4 p, 2 p, 2 p
    small_inv<0, 0>(y, tw, lane, q, off4);
    small_inv<0, 1>(y, tw, lane, q, off_b);
    y[0] = reduce_to(y[0], 16, 2, q);
    y[4] = reduce_to(y[4], 16, 2, q);
    small_inv<0, 2>(y, tw, lane, q, off_c);
    y[1] = reduce_to(y[1], 8, 4, q);
    small_exchange<1, 0, 3>(x, buf, lane);
    small_inv<3, 3>(y, tw, lane, q, off4);
    small_inv<3, 4>(y, tw, lane, q, off_b);
    y[0] = reduce_to(y[0], 16, 2, q);
    y[4] = reduce_to(y[4], 16, 2, q);
    small_inv<3, 5>(y, tw, lane, q, off_c);
    y[1] = reduce_to(y[1], 8, 4, q);
    small_exchange<1, 3, 5>(x, buf, lane);
    small_inv<5, 6>(y, tw, lane, q, off4);
    small_inv<5, 7>(y, tw, lane, q, [&](int c) { return (c & 2) ? q.p2 : q.p8; });
    y[0] = reduce_to(y[0], 16, 4, q);
    y[1] = reduce_to(y[1], 16, 4, q);
}

template <int MAXK, int MINB>
__global__ void __launch_bounds__(64 * (MAXK + 1), MINB)
bootstrap_small_kernel(LaunchShape S, DeviceKeys K, const GateDesc *__restrict__ desc,
                       const uint32_t *__restrict__ ct_a, const uint32_t *__restrict__ ct_b,
                       const uint32_t *__restrict__ abar_in, int64_t max_steps, uint32_t *__restrict__ ext,
                       uint32_t *__restrict__ acc_out) {
    constexpr int N = kSmallN, UNITS = N / 4;  // 16-byte units of a key plane
    extern __shared__ __align__(16) unsigned char smem[];
    const int k = (int)S.k, n = (int)S.n, threads = 64 * (k + 1);
    const SmallLayout L = small_layout(S.k, S.n);
    const int wid = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31, jj = wid >> 1, pr = wid & 1, bar = 1 + jj, t64 = threadIdx.x & 63;
    const uint2 *tw_f = reinterpret_cast<const uint2 *>(smem + L.tw) + pr * N, *tw_i = tw_f + 2 * N;
    uint32_t *acc = reinterpret_cast<uint32_t *>(smem + L.acc) + jj * N;
    uint32_t *buf = reinterpret_cast<uint32_t *>(smem + L.xbuf) + wid * 3 * kSmallX;
    uint32_t *buf_other = reinterpret_cast<uint32_t *>(smem + L.xbuf) + (wid ^ 1) * 3 * kSmallX;
    uint32_t *shares = reinterpret_cast<uint32_t *>(smem + L.shares);
    uint32_t *vbuf = reinterpret_cast<uint32_t *>(smem + L.vbuf) + jj * N;
    uint16_t *abar = reinterpret_cast<uint16_t *>(smem + L.abar);
    {
        const uint4 *src = static_cast<const uint4 *>(K.tw_split);
        uint4 *dst = reinterpret_cast<uint4 *>(smem + L.tw);
        for (int x = threadIdx.x; x < 4 * N / 2; x += threads) dst[x] = src[x];
    }
    if (abar_in) {
        const uint32_t W = S.k * S.n + 1;
        for (uint32_t x = threadIdx.x; x < W; x += threads) abar[x] = (uint16_t)abar_in[(size_t)blockIdx.x * W + x];
    } else {
        lin_modswitch(S, desc[blockIdx.x], ct_a, ct_b, abar, threadIdx.x, threads);
    }
    __syncthreads();
    const PrimeK q = prime_of(pr, S.d - 3);
    const Gadget gad = make_gadget(8);
    {
        const uint32_t bbar = abar[k * n];
        for (uint32_t m = t64; m < (uint32_t)N; m += 64) {
            const uint32_t r = (m + bbar) & (2 * N - 1);
            acc[m] = jj ? 0u : ((r >= (uint32_t)N) ? (0u - (1u << 29)) : (1u << 29));
        }
    }
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;\n" ::"r"(bar) : "memory"); };
    pair_sync();
    // key words of this lane's elements 8 lane .. 8 lane + 7
    const int u0 = 2 * lane, pos0 = (u0 & 7) * (N / 32) + ((u0 >> 3) ^ (u0 & 7)),
              pos1 = ((u0 + 1) & 7) * (N / 32) + ((u0 >> 3) ^ ((u0 + 1) & 7));
    auto load_key8 = [&](uint32_t(&key)[3][8], const uint4 *src) {  // three polynomials of a key
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const uint4 a = __ldg(src + l * 2 * UNITS + pos0), b = __ldg(src + l * 2 * UNITS + pos1);
            key[l][0] = a.x, key[l][1] = a.y, key[l][2] = a.z, key[l][3] = a.w;
            key[l][4] = b.x, key[l][5] = b.y, key[l][6] = b.z, key[l][7] = b.w;
        }
    };
    const uint4 *bk_all = static_cast<const uint4 *>(K.bk) + pr * UNITS;
    uint32_t ka[3][8];
    load_key8(ka, static_cast<const uint4 *>(K.keyA) + (size_t)jj * 6 * UNITS + pr * UNITS);
    // Integers (mod 2^32) of coefficients lane + 32 (4 pr + c) from both primes' residues (below 4 p).
    auto recombine = [&](uint32_t(&y)[8], uint32_t(&z)[4]) {
#pragma unroll
        for (int c = 0; c < 4; ++c) buf[32 * c + lane] = pr ? y[c] : y[4 + c];
        pair_sync();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t own = pr ? y[4 + c] : y[c], other = buf_other[32 * c + lane];
            z[c] = crt_centred(pr ? other : own, pr ? own : other);
        }
        pair_sync();  // both buffers have been read
    };
    auto cut = [&](uint32_t(&x)[3][8], int c, uint32_t word) {
#pragma unroll
        for (int l = 0; l < 3; ++l) x[l][c] = q.p + ((word >> (24 - 8 * l)) & 255u) - 128u;
    };

    const int all_steps = k * n;
    const int limit = (max_steps >= 0 && max_steps < all_steps) ? (int)max_steps : all_steps;
    int i = 1, left = n;
    uint32_t parity = 0, e_next = abar[0];
#pragma unroll 1
    for (int step = 0; step < limit; ++step) {
        const uint32_t e = e_next;
        e_next = abar[step + 1];
        if (left == 0) {
            left = n;
            ++i;
        }
        --left;
        if (e == 0) continue;  // X^0 - 1 = 0: the product adds nothing
        const uint4 *bk = bk_all + (size_t)step * 18 * UNITS;
        const bool last = jj == 0 || jj == i;
        uint32_t x[3][8], key[3][8], C[8];
        load_key8(key, bk);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint32_t m = lane + 32 * c, r = m + e;
            const uint32_t a = acc[r & (N - 1)];
            const uint32_t neg = (uint32_t)((int32_t)(r << 23) >> 31);  // bit 8 of r: -1
            cut(x, c, (a ^ neg) - neg - acc[m] + gad.offset);
        }
        small_forward<3>(x, tw_f, buf, lane, q);
        {
            uint32_t V[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                C[c] = mac3_redc(x[0][c], x[1][c], x[2][c], key[0][c], key[1][c], key[2][c], q);
                V[c] = mac3_redc(x[0][c], x[1][c], x[2][c], ka[0][c], ka[1][c], ka[2][c], q);
            }
            uint4 *dst = reinterpret_cast<uint4 *>(shares + ((parity * (k + 1) + jj) * 2 + pr) * N) + lane;
            dst[0] = make_uint4(V[0], V[1], V[2], V[3]);
            dst[32] = make_uint4(V[4], V[5], V[6], V[7]);
        }
        if (last) load_key8(key, bk + (jj == 0 ? 6 : 12) * UNITS);
        __syncthreads();  // every share is stored
        uint32_t y[1][8], z[4];
        if (last) {
            const uint4 *src = reinterpret_cast<const uint4 *>(shares + (parity * (k + 1) * 2 + pr) * N) + lane;
            auto take = [&](const uint4 &a, int at, bool first) {
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const uint32_t t = (first ? 0u : y[0][at + h]) + word_of(a, h);  // each below 4 p
                    y[0][at + h] = first ? t : min(t, t - q.p4);
                }
            };
            take(src[0], 0, true);
            take(src[32], 4, true);
            for (int s = 1; s <= k; ++s) {
                take(src[s * 2 * UNITS], 0, false);
                take(src[s * 2 * UNITS + 32], 4, false);
            }
            small_inverse(y, tw_i, buf, lane, q);
            recombine(y[0], z);
#pragma unroll
            for (int c = 0; c < 4; ++c) vbuf[lane + 32 * (4 * pr + c)] = z[c] + gad.offset;
            pair_sync();
#pragma unroll
            for (int c = 0; c < 8; ++c) cut(x, c, vbuf[lane + 32 * c]);
            small_forward<3>(x, tw_f, buf, lane, q);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint32_t a = C[c] + mac3_redc(x[0][c], x[1][c], x[2][c], key[0][c], key[1][c], key[2][c], q);
                C[c] = min(a, a - q.p4);
            }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) y[0][c] = C[c];
        small_inverse(y, tw_i, buf, lane, q);
        recombine(y[0], z);
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[lane + 32 * (4 * pr + c)] += z[c];
        pair_sync();
        parity ^= 1;
    }
    if (acc_out) {
        uint32_t *dst = acc_out + ((size_t)blockIdx.x * (k + 1) + jj) * N;
        for (uint32_t x = t64; x < (uint32_t)N; x += 64) dst[x] = acc[x];
    } else {
        uint32_t *dst = ext + (size_t)blockIdx.x * (k * N + 1);
        if (jj == 0) {
            if (t64 == 0) dst[k * N] = acc[0] + (1u << 29);  // +1/8
        } else {
            for (int m = t64; m < N; m += 64) dst[(jj - 1) * N + m] = m == 0 ? acc[0] : 0u - acc[N - m];
        }
    }
}

}  // namespace br
}  // namespace mk
