// mk_keyswitch_tc.cu -- the key switch as an exact matrix product on tcgen05.
//
// MKKeySwitch (Sec. 3.2 of arXiv 2205.05825) adds, for every party i,
// coefficient j and digit position l, the row KS_i[j][l][delta - 1] its 2-bit
// digit delta != 0 selects.  Over a batch of gates that is a product of 0/1
// indicators with the key rows:
//   out[g][x] = sum_(j, l, e) [delta_g(j, l) = e] KS[j][l][e - 1][x],
// K = 24 per coefficient.  The key words are cut into three unsigned planes
// of 11, 11 and 10 bits, exact in fp16 as the indicators are; each digit
// selects at most one of its three rows, so a party's sum of a plane is at
// most 8 N 2047 < 2^24 for N <= 1024 and fp32 accumulation in TMEM is exact.
//
// What bounded the SIMT kernels: the batched one reads a shared-memory slot
// per gate, digit and column (4 bytes each: 37.6 G reads at 4096 gates, k = 2)
// and ran one CTA per 32 gates and 128 columns over the whole K range, so a
// small batch kept 15 CTAs busy for 8 ms; the one-gate kernel walked 16 k
// dependent row reads a thread.  Here a work item is 256 (or 128) gates x 85
// output words (255 of 256 MMA columns, word x plane interleaved) x one party
// x one of `splits` K ranges, and items add into the output rows with
// 32-bit reductions (integer sums: any order gives the same words).  Split-K
// fills the chip whatever the batch.
//
// A CTA: warps 0-7 build the indicator tiles (one gate per thread; digit
// words staged 32 coefficients at a time by coalesced reads of the gate's
// row) and drain TMEM at the end; warp 8 bulk-copies the key tiles, laid out
// in HBM as the operand blocks (24 KB per coefficient pair and column tile);
// warp 9 issues the MMAs.  Four stages of a coefficient pair (K = 48) each.
// Every wait is bounded in global time (S.wait_ns): one that runs out sets
// the CTA's abort word and the context's status word, every role leaves at
// its next wait, the copies and MMAs in flight are waited for (bounded), and
// mk_sync reports MK_ETIMEOUT.
#include <cuda_fp16.h>

#include "mk_bulk.cuh"
#include "mk_internal.h"

namespace mk {
namespace {

using br::st_bulk_load;
using br::st_fence_proxy_async;
using br::st_globaltimer;
using br::st_mbar_init;
using br::st_mbar_try;
using br::st_smem_addr;

constexpr uint32_t KT_WORDS = 85;            // output words of a column tile
constexpr uint32_t KT_BBLOCK = 6 * 256 * 16;  // one coefficient pair of a key tile: 6 K units x 256 rows x 16 bytes
constexpr uint32_t KT_AHALF = 6 * 128 * 16;   // indicators of 128 gates
constexpr uint32_t KT_STAGE = KT_BBLOCK + 2 * KT_AHALF;
constexpr int KT_STAGES = 4;
constexpr int KT_BUILDERS = 256, KT_THREADS = KT_BUILDERS + 64;
constexpr uint32_t KT_CHUNK = 32;            // coefficients staged at a time
constexpr uint32_t KT_PITCH = 258;           // halves per staged coefficient (bank shift of one word)
constexpr uint64_t KT_DRAIN_NS = 1000000000ull;
// kind::f16: fp32 accumulator, fp16 operands, both K-major, N = 256, M = 128
constexpr uint32_t KT_IDESC = (1u << 4) | ((256u >> 3) << 17) | ((128u >> 4) << 24);

struct KtCtl {
    unsigned long long full[KT_STAGES], ready[KT_STAGES], empty[KT_STAGES], done;
    uint32_t tmem, abort;
};
constexpr size_t KT_OFF_WORDS = (size_t)KT_STAGES * KT_STAGE;
constexpr size_t KT_OFF_CTL = KT_OFF_WORDS + ((KT_CHUNK * KT_PITCH * 2 + 15) & ~15u);
constexpr size_t KT_SMEM = KT_OFF_CTL + sizeof(KtCtl);
static_assert(KT_SMEM <= 227 * 1024, "shared memory of a CTA");

// Wait for the phase of parity `parity`; false if the bound or another role's
// abort ended it.  abort == nullptr: only the bound (the CTA's own copies and MMAs).
__device__ __noinline__ bool kt_wait(uint32_t bar, uint32_t parity, uint64_t wait_ns, volatile uint32_t *abort) {
    if (st_mbar_try(bar, parity)) return true;
    const uint64_t t0 = st_globaltimer();
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        if (st_mbar_try(bar, parity)) return true;
        if (abort && *abort) return false;
        if (st_globaltimer() - t0 > wait_ns) break;
    }
    if (abort) *abort = 1u;
    return false;
}

__device__ __forceinline__ uint64_t kt_desc(uint32_t saddr, uint32_t k_stride) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(k_stride >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) |
           (1ull << 46);
}

__device__ __forceinline__ void kt_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// Indicators [delta = e] of the eight digits in the 16-bit word: `bits` has a
// one at bit 2 (7 - l) for every digit l that equals e.  Half 2 t stands for
// digit t + 4, half 2 t + 1 for digit t: their bits are 8 apart, so one byte
// permutation by the two bits builds both halves (1.0 = 0x3C00).
__device__ __forceinline__ uint4 kt_indicators(uint32_t bits) {
    return make_uint4(__byte_perm(0x3C00u, 0, (bits >> 2) & 0x1010u), __byte_perm(0x3C00u, 0, bits & 0x1010u),
                      __byte_perm(0x3C00u, 0, (bits << 2) & 0x1010u), __byte_perm(0x3C00u, 0, (bits << 4) & 0x1010u));
}

// columns [c, c + 16) of this warp's TMEM lanes
__device__ __forceinline__ void kt_ld16(uint32_t addr, float *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
          "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
        : "r"(addr));
}

// Blocks: column tile fastest, then party, then K range, then group of 128 MT gates (all on grid.x: grid.y would end
// at 65535 groups, 16.8 M rows).
template <int MT>
__global__ void __launch_bounds__(KT_THREADS, 1)
    keyswitch_tc_kernel(LaunchShape S, const unsigned char *__restrict__ planes, const GateDesc *__restrict__ desc,
                        const uint32_t *__restrict__ ext, uint32_t *__restrict__ out, uint32_t count, uint32_t tiles,
                        uint32_t splits, uint32_t *status) {
    extern __shared__ __align__(128) unsigned char smem[];
    KtCtl *ctl = reinterpret_cast<KtCtl *>(smem + KT_OFF_CTL);
    uint16_t *words = reinterpret_cast<uint16_t *>(smem + KT_OFF_WORDS);
    const uint32_t n = S.n, N = S.N, k = S.k;
    const uint32_t E = k * N + 1, W = k * n + 1;
    const uint32_t items = tiles * k * splits, item = blockIdx.x % items;
    const uint32_t tile = item % tiles, party = item / tiles % k, split = item / tiles / k;
    const uint32_t g0 = blockIdx.x / items * (128 * MT);
    const uint32_t chunks = N / KT_CHUNK, c0 = split * chunks / splits, c1 = (split + 1) * chunks / splits;
    const uint32_t kb0 = c0 * (KT_CHUNK / 2), nkb = (c1 - c0) * (KT_CHUNK / 2);  // coefficient pairs of this item
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile uint32_t *abort = &ctl->abort;
    const uint32_t stage0 = st_smem_addr(smem);
    const uint32_t full0 = st_smem_addr(&ctl->full[0]), ready0 = st_smem_addr(&ctl->ready[0]),
                   empty0 = st_smem_addr(&ctl->empty[0]), done = st_smem_addr(&ctl->done);

    if (tid == 0) {
        for (int s = 0; s < KT_STAGES; ++s) {
            st_mbar_init(full0 + 8 * s, 1);
            st_mbar_init(ready0 + 8 * s, 4 * MT);
            st_mbar_init(empty0 + 8 * s, 1);
        }
        st_mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        ctl->abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(st_smem_addr(&ctl->tmem)),
                     "r"(256u * MT)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = ctl->tmem;
    bool ok = true;

    if (warp == 8) {
        if (lane == 0) {
            const unsigned char *src = planes + ((size_t)(party * (N / 2) + kb0) * tiles + tile) * KT_BBLOCK;
            uint32_t kb = 0;
            for (; kb < nkb; ++kb) {
                const uint32_t st = kb % KT_STAGES;
                if (kb >= KT_STAGES && !kt_wait(empty0 + 8 * st, (kb / KT_STAGES - 1) & 1, S.wait_ns, abort)) {
                    ok = false;
                    break;
                }
                if (kb0 + kb == S.skip_key_tile) continue;  // test hook
                st_bulk_load(stage0 + st * KT_STAGE, src + (size_t)kb * tiles * KT_BBLOCK, KT_BBLOCK, full0 + 8 * st);
            }
            // no copy may be in flight when the CTA exits
            for (uint32_t q = kb > KT_STAGES ? kb - KT_STAGES : 0; q < kb; ++q)
                if (kb0 + q != S.skip_key_tile) kt_wait(full0 + 8 * (q % KT_STAGES), (q / KT_STAGES) & 1, KT_DRAIN_NS, nullptr);
        }
        __syncwarp();
    } else if (warp == 9) {
        if (lane == 0) {
            for (uint32_t kb = 0; kb < nkb; ++kb) {
                const uint32_t st = kb % KT_STAGES, ph = (kb / KT_STAGES) & 1;
                ok = kt_wait(full0 + 8 * st, ph, S.wait_ns, abort) && kt_wait(ready0 + 8 * st, ph, S.wait_ns, abort);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const uint64_t bd = kt_desc(stage0 + st * KT_STAGE, 4096);
                const uint64_t ad = kt_desc(stage0 + st * KT_STAGE + KT_BBLOCK, 2048);
#pragma unroll
                for (int ks = 0; ks < 3; ++ks)
#pragma unroll
                    for (int m = 0; m < MT; ++m)
                        asm volatile(
                            "{\n\t.reg .pred p;\n\t"
                            "setp.ne.b32 p, %4, 0;\n\t"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem + 256 * m),
                            "l"(ad + (m * KT_AHALF + ks * 4096) / 16), "l"(bd + ks * 8192 / 16), "r"(KT_IDESC),
                            "r"(kb | (uint32_t)ks));
                kt_commit(empty0 + 8 * st);
            }
            kt_commit(done);  // every MMA of this thread
            kt_wait(done, 0, KT_DRAIN_NS, nullptr);  // whatever became of the builders' wait for it
        }
        __syncwarp();
    } else if (warp < 4 * MT) {
        // Builder of gate g0 + tid
        const uint32_t round_off = 1u << 15;  // 16 digit bits
        unsigned char *a_row = smem + KT_BBLOCK + (tid >> 7) * KT_AHALF + (tid & 127) * 16;
        uint32_t kb = 0;
        for (uint32_t c = c0; c < c1 && ok; ++c) {
            __syncwarp();  // this warp's words of the previous chunk are consumed
            const uint32_t *src = ext + (size_t)party * N + c * KT_CHUNK + lane;
#pragma unroll 8
            for (int q = 0; q < 32; ++q) {
                const uint32_t g = g0 + 32 * warp + q;
                const uint32_t v = g < count ? __ldg(src + (size_t)g * E) + round_off : 0u;
                words[lane * KT_PITCH + 32 * warp + q] = (uint16_t)(v >> 16);
            }
            __syncwarp();
            const bool live = g0 + tid < count;
            for (uint32_t b = 0; b < KT_CHUNK / 2; ++b, ++kb) {
                const uint32_t st = kb % KT_STAGES;
                if (kb >= KT_STAGES && !kt_wait(empty0 + 8 * st, (kb / KT_STAGES - 1) & 1, S.wait_ns, abort)) ok = false;
                if (!__all_sync(0xFFFFFFFFu, ok)) {
                    ok = false;
                    break;
                }
                uint4 *dst = reinterpret_cast<uint4 *>(a_row + st * KT_STAGE);
#pragma unroll
                for (int jj = 0; jj < 2; ++jj) {
                    const uint32_t x = live ? words[(2 * b + jj) * KT_PITCH + tid] : 0u;
                    const uint32_t lo = x & 0x5555u, hi = (x >> 1) & 0x5555u;
                    dst[(3 * jj) * 128] = kt_indicators(lo & ~hi);
                    dst[(3 * jj + 1) * 128] = kt_indicators(hi & ~lo);
                    dst[(3 * jj + 2) * 128] = kt_indicators(hi & lo);
                }
                st_fence_proxy_async();
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(ready0 + 8 * st) : "memory");
            }
        }
        if (ok) ok = kt_wait(done, 0, S.wait_ns, abort);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (ok) {
            // lane = gate: integer words through this warp's part of the (now free) stages, then rows of 85 words
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            uint32_t *buf = reinterpret_cast<uint32_t *>(smem) + warp * (32 * KT_WORDS);
            const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + 256 * (warp >> 2);
#pragma unroll 1
            for (int c = 0; c < 6; ++c) {
                float f[48];
                kt_ld16(ta + 48 * c, f);
                if (c < 5) {
                    kt_ld16(ta + 48 * c + 16, f + 16);
                    kt_ld16(ta + 48 * c + 32, f + 32);
                }
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                for (int x = 0; x < 16; ++x)
                    if (c < 5 || x < 5)
                        buf[lane * KT_WORDS + 16 * c + x] = __float2uint_rn(f[3 * x]) +
                                                            (__float2uint_rn(f[3 * x + 1]) << 11) +
                                                            (__float2uint_rn(f[3 * x + 2]) << 22);
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            const uint32_t x0 = tile * KT_WORDS;
            for (int q = 0; q < 32; ++q) {
                const uint32_t g = g0 + 32 * warp + q;
                if (g >= count) break;
                uint32_t *row = out + (size_t)(desc ? desc[g].out : g) * W;
                for (uint32_t x = lane; x < KT_WORDS && x0 + x <= n; x += 32)
                    atomicAdd(row + (x0 + x < n ? party * n + x0 + x : k * n), buf[q * KT_WORDS + x]);
            }
        }
    }
    if (!__syncthreads_and(ok) && tid == 0) atomicOr(status, kStatusKeyswitch);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(256u * MT) : "memory");
}

// Output rows before the items add into them: zero masks, b from the extracted sample.
__global__ void keyswitch_init_kernel(LaunchShape S, const GateDesc *__restrict__ desc, const uint32_t *__restrict__ ext,
                                      uint32_t *__restrict__ out) {
    const uint32_t W = S.k * S.n + 1, g = blockIdx.x;
    uint32_t *row = out + (size_t)(desc ? desc[g].out : g) * W;
    for (uint32_t x = threadIdx.x; x < W; x += blockDim.x)
        row[x] = x == W - 1 ? ext[(size_t)g * (S.k * S.N + 1) + S.k * S.N] : 0u;
}

// One block per (party, coefficient pair, column tile): thread r holds row r
// (word r / 3, plane r % 3) of the operand block's six K units.
__global__ void keyswitch_planes_kernel(LaunchShape S, const uint32_t *__restrict__ ks, uint4 *__restrict__ planes,
                                        uint32_t tiles) {
    const uint32_t n = S.n, tile = blockIdx.x % tiles, pair = blockIdx.x / tiles;  // pair: party * N / 2 + j / 2
    const uint32_t r = threadIdx.x, x = tile * KT_WORDS + r / 3, pl = r % 3;
    const bool live = r < 3 * KT_WORDS && x <= n;
    uint4 *dst = planes + (size_t)blockIdx.x * (KT_BBLOCK / 16) + r;
    for (uint32_t u = 0; u < 6; ++u) {
        const uint32_t j = 2 * pair + u / 3, e = u % 3;
        uint32_t h[8];
#pragma unroll
        for (uint32_t i = 0; i < 8; ++i) {
            const uint32_t l = (i & 1) ? i / 2 : i / 2 + 4;
            const uint32_t w = live ? ks[(((size_t)j * 8 + l) * 3 + e) * (n + 1) + x] : 0u;
            const uint32_t v = pl == 0 ? w & 2047u : (pl == 1 ? (w >> 11) & 2047u : w >> 22);
            h[i] = __half_as_ushort(__uint2half_rn(v));
        }
        dst[u * 256] = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
    }
}

uint32_t column_tiles(const LaunchShape &S) { return (S.n + 1 + KT_WORDS - 1) / KT_WORDS; }
}  // namespace

bool keyswitch_tc_supported(const LaunchShape &S) {
    return S.ks_bit == 2 && S.t == 8 && S.N % KT_CHUNK == 0 && S.N <= 1024;
}

size_t keyswitch_planes_bytes(const LaunchShape &S) {
    return keyswitch_tc_supported(S) ? (size_t)S.k * (S.N / 2) * column_tiles(S) * KT_BBLOCK : 0;
}

cudaError_t build_keyswitch_planes(const LaunchShape &S, const uint32_t *ks, void *planes, cudaStream_t st) {
    if (!keyswitch_tc_supported(S)) return cudaErrorInvalidValue;
    const uint32_t tiles = column_tiles(S);
    keyswitch_planes_kernel<<<S.k * (S.N / 2) * tiles, 256, 0, st>>>(S, ks, static_cast<uint4 *>(planes), tiles);
    return cudaGetLastError();
}

cudaError_t launch_keyswitch_tc(const LaunchShape &S, const DeviceKeys &K, const GateDesc *desc, const uint32_t *ext,
                                uint32_t *out, uint32_t count, cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    if (!keyswitch_tc_supported(S) || !K.ks_planes || !K.status) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const uint32_t tiles = column_tiles(S), mt = count > 128 ? 2 : 1, groups = (count - 1) / (128 * mt) + 1;
    // K ranges per item: the fewest waves x (a fixed cost of about 8 us + the range's pairs at the slower of the
    // MMAs, 0.19 us per 128 gates, and the key copy, 0.3 us)
    uint32_t splits = 1;
    double best = 1e30;
    for (uint32_t s = 1; s <= S.N / KT_CHUNK; s *= 2) {
        const uint64_t waves = ((uint64_t)tiles * S.k * groups * s + sms - 1) / sms;
        const double us = (double)waves * (8.0 + (S.N / 2 / s) * (mt == 2 ? 0.38 : 0.3));
        if (us < best) {
            best = us;
            splits = s;
        }
    }
    const uint64_t grid = (uint64_t)tiles * S.k * splits * groups;
    if (grid > 0x7FFFFFFFu || count > 0x7FFFFFFFu) return cudaErrorInvalidConfiguration;  // before any row is written
    keyswitch_init_kernel<<<count, 256, 0, st>>>(S, desc, ext, out);
    auto run = [&](auto kern) {
        cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)KT_SMEM);
        if (err != cudaSuccess) return err;
        kern<<<(uint32_t)grid, KT_THREADS, KT_SMEM, st>>>(S, static_cast<const unsigned char *>(K.ks_planes), desc, ext, out, count,
                                                tiles, splits, K.status);
        return cudaGetLastError();
    };
    return mt == 2 ? run(keyswitch_tc_kernel<2>) : run(keyswitch_tc_kernel<1>);
}

}  // namespace mk
