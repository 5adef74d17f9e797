// mk_bootstrap_warp.cuh -- the two-prime blind rotation with two warps per
// (gate, prime), tcgen05 for the first six stages of every forward transform
// and register-resident butterflies for the rest (N = 1024, base 2^8, d = 3).
//
// The batched kernel of mk_bootstrap.cuh is bound by waits: four passes over
// 8 elements a thread need three shared-memory exchanges with CTA barriers
// per transform, and the multiplies of its butterflies (Shoup: one high and
// two low multiplies, 8 cycles of a scheduler's 16-lane multiply pipe per
// warp) bound it from below at about 12.5 k clocks per CMux step of a gate at
// k = 2.  Here
//  * coefficient m is u[c + 16 s], 16 columns x 64 rows.  Reducing a
//    polynomial modulo the 64 factors X^16 - zeta_y of X^1024 + 1 mod p (the
//    state of the transform after six of its ten stages) is, for digits, a
//    product of a constant 64 x 64 matrix with small integers: y_y[c] =
//    sum_s zeta_y^s u[c + 16 s].  zeta_y^s is cut into three signed planes of
//    9, 9 and 10 bits, exact in fp16 as the digits are.  One tcgen05.mma
//    sequence per plane (M = 128: both primes' 64 factors; N = 48: the three
//    digit polynomials' columns; K = 64) sums it exactly in fp32 in TMEM.  A
//    last K step of constants starts every sum at 1.5 2^23, so the sums' bit
//    patterns are the integers; two FMAs estimate the quotient by p and three
//    multiply-adds recombine the planes.  TMEM lane = (prime, factor), so
//    tcgen05.ld hands each thread the 16 elements of its factor: no
//    transposition through shared memory;
//  * the last four stages run in registers without a barrier, for the three
//    digit polynomials together (they share the lane's 15 twiddles).  No value
//    is reduced on the way: it starts below 3.6 p and grows by 2 p a stage
//    (16 p < 2^32);
//  * the inverse runs four stages in the factors, transposes within the warp,
//    runs four more, and the last two follow an exchange among the gate's
//    four warps that also brings the two primes' residues together for the
//    recombination (CRT).  Bounds are tracked at compile time and a value is
//    reduced only where a sum could pass 2^32;
//  * the lane that ends with a coefficient is the one that cuts its next
//    digits: eight coefficients of a lane are one 16-byte unit of the matrix
//    operand, so v's digits need no further exchange.
//  The four warps meet at a 128-thread barrier; gates of a CTA run
//  independently of each other.  A slot's matrix products are started as soon
//  as the one before it has left TMEM, so they run under its butterflies; the
//  first group of a slot's key words is loaded before them (two groups ahead
//  measured slower: it spills).
//
// (The same matrix product by warp-level mma.sync gave 18.0 k clocks per CMux
// step of a gate: on this chip it competes with the integer multiplies for
// the register file, and its fragments need a transposition.)
//
// Measured (GB300, whole blind rotation): 4096 gates at k = 2 347 -> 211 ms,
// 1001 at k = 4 308 -> 184 ms (170 with the last pass in another kernel,
// bootstrap_head), 152 at k = 2 (one gate per SM) 31 -> 14.3 ms.  Per CMux step and gate 23.7 -> 14.5 k clocks of an SM;
// the multiply pipe is 81 % busy (ncu, three gates an SM).
//
// A CTA holds G gates (4 G warps) and the tables once; the grid is at most one
// CTA per SM and walks the gates with stride G * gridDim.
// Exact: the same integers as every other exact form, hence the same
// ciphertexts (hybrid product as in mk_bootstrap.cuh; arXiv 2205.05825,
// Sec. 3.2 and 4.1).
#pragma once
#include <cstddef>

#include <cuda_fp16.h>

#include "mk_bootstrap.cuh"
#include "mk_bulk.cuh"

namespace mk {
namespace br {

// Constants of one prime.
struct PrimeK {
    uint32_t p, p2, p4, p8;
    uint32_t zero;        // 0, unknown to the compiler: a sum of three stays off the multiply pipe
    uint32_t pinv;        // p^-1 mod 2^32
    float c1, c2, kf;     // quotient estimate fma(f2, c2, fma(f1, c1, kf))
};

// The planes' sums come as f_i = m_i + s_i (m_1 = m_2 = M = 1.5 2^23, bits
// 0x4B400000 + s_i), and y = s_0 + 2^9 s_1 + 2^18 s_2 - q p + 2 p is wanted
// from bits(f_0) + 2^9 bits(f_1) + 2^18 bits(f_2) - bits(qf) p mod 2^32 alone,
// qf = M + q + A.  With m_0 = M + B that holds if B - A p = 2 p -
// M' (1 + 2^9 + 2^18) + M' p mod 2^32 (M' = 0x4B400000); small solutions keep both
// floats in [2^23, 2^24).
template <uint32_t Pm, uint32_t PINV, int A, int B>
__device__ __forceinline__ PrimeK prime_k() {
    constexpr uint32_t bits = 0x4B400000u;
    static_assert((uint32_t)B == 2u * Pm - bits * (1u + 512u + 262144u) + bits * Pm + (uint32_t)A * Pm, "plane offsets");
    static_assert(A < (1 << 20) && A > -(1 << 20) && B < (1 << 15) && B > -(1 << 15), "plane offsets");
    constexpr double magic = 12582912.0, c1 = 512.0 / Pm, c2 = 262144.0 / Pm;
    constexpr long long kf = (long long)(magic - magic * (c1 + c2) + 0.5) + A;
    PrimeK q;
    q.p = Pm;
    q.p2 = 2 * Pm;
    q.p4 = 4 * Pm;
    q.p8 = 8 * Pm;
    q.pinv = 0u - PINV;
    q.c1 = (float)c1;
    q.c2 = (float)c2;
    q.kf = (float)kf;
    return q;
}
__device__ __forceinline__ PrimeK prime_of(int pr, uint32_t zero) {
    PrimeK q = pr ? prime_k<P2, PINV2, 3639, -4551>() : prime_k<P1, PINV1, 245762, -16380>();
    q.zero = zero;
    return q;
}

// ---------------------------------------------------------------- tables
// Global block of the tables, copied whole into shared memory (uint4 units):
//   halves [2 primes][2 h][8][32 lanes]: unit u of lane x holds entries 2u, 2u + 1
//     of the heap of 16 {w, w'} of half row y = 32 h + x (elements 16 y ..
//     16 y + 15 of the transform): entry b + i (b = 1, 2, 4, 8; i < b) is the
//     forward twiddle 64 b + b y + i (entry 0 unused);
//   rows [2][16]: entries 2u, 2u + 1 of forward twiddles 32 .. 63 (stage six of row f);
//   cross [2][16]: entries 2u, 2u + 1 of forward twiddles 0 .. 31 (0 unused);
//   ones: the B operand's constant K step (48 columns): 4096, 64, 1, zeros;
//   planes [3][4 K steps][2 units][128 rows]: A operand (fp16, 8 K slots a
//     unit): the planes of zeta_y^s, row 64 prime + y; K slot 8 a + i stands for
//     s = 2 a + 16 (i / 2) + i % 2;
//   start [2][128 rows]: unit 0 of the A operand's constant K step (its unit 1
//     is zero): 3072, then the offset B of plane 0 as 64 b1 + b0, or 0 for
//     planes 1 and 2.
// The first four blocks and, where TMEM has no room for it, plane 0 are copied
// into shared memory; the rest of the A operand goes into TMEM (rows = lanes,
// two K slots a column), where the tensor core reads it without competing for
// shared memory: with all of it there a step's products took 15 x 5.6 KB of
// shared-memory reads.  Operand blocks in shared memory are K-major without
// swizzle: 8 rows x 16 bytes contiguous, row groups 128 bytes apart, K units
// of A 2048 and of B 768 bytes apart.
constexpr int kTabHalves = 2 * 2 * 8 * 32, kTabRows = 2 * 16, kTabCross = 2 * 16, kTabOnes = 2 * 48;
constexpr int kTabPlane = 4 * 256, kTabStart = 2 * 128;
constexpr int kTabSmall = kTabHalves + kTabRows + kTabCross + kTabOnes;
constexpr int kTabUnits = kTabSmall + 3 * kTabPlane + kTabStart;
static_assert(kTabUnits * 16 == kWarpTableBytes, "table block");
constexpr uint32_t kAUnit = 2048, kBUnit = 768;  // K-unit strides in bytes

// A CTA with D gates (or teams): 144 TMEM columns each, then the constant
// steps (8 columns each) and the planes (32 each), plane 0 in shared memory if
// D = 3.
template <int D>
struct Operands {
    static constexpr int first = D == 3 ? 1 : 0;  // first plane in TMEM
    static constexpr uint32_t start = 144 * D, planes = start + 16, used = planes + 32 * (3 - first);
    static constexpr uint32_t columns = used <= 256 ? 256 : 512;
    static constexpr int units = kTabSmall + first * kTabPlane;  // table units in shared memory
    static_assert(used <= 512, "TMEM columns");
};

// ---------------------------------------------------------------- shared memory
// A control block, then per gate: accumulators, digits (the B operand, 6 KB),
// the warps' transposition buffers (2 KB each; together the exchange buffer),
// c'_0 between its slot and v's, the mod-switched words.
constexpr int kWarpMaxGates = 3;  // 144 TMEM columns each
struct WarpCtl {
    unsigned long long bar[kWarpMaxGates];  // mbarriers: a gate's matrix products
    uint32_t tmem, abort;
};
struct WarpLayout {
    size_t ctl, gate, gate_bytes, total;
    size_t acc, digits, xbuf, park, abar;
};

__host__ __device__ inline WarpLayout warp_layout(uint32_t k, uint32_t n, uint32_t gates) {
    WarpLayout L;
    L.ctl = (size_t)Operands<kWarpMaxGates>::units * 16;
    L.gate = L.ctl + ((sizeof(WarpCtl) + 15) & ~size_t(15));
    L.acc = 0;
    L.digits = L.acc + (size_t)4096 * (k + 1);
    L.xbuf = L.digits + 8 * kBUnit;
    L.park = L.xbuf + 8192;
    L.abar = L.park + 8192;
    L.gate_bytes = L.abar + ((sizeof(uint16_t) * (k * n + 1) + 15) & ~size_t(15));
    L.total = L.gate + L.gate_bytes * gates;
    return L;
}

// Lets a kernel have all of an SM's shared memory.  The limit is the kernel's,
// not the launch's: set to what each launch needs, a smaller one from another
// thread (other gates a CTA, or another context's k and n) could come between
// a thread's setting and its launch, which would then be refused.
template <class Kernel>
cudaError_t allow_smem(Kernel kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWarpSmemMax);
}

__device__ __forceinline__ void quad_sync(int bar) { asm volatile("bar.sync %0, 128;\n" ::"r"(bar) : "memory"); }

// Accumulator polynomials: coefficient m at m ^ 16 (m / 32 mod 2), so that a
// warp's reads of 16 columns x 2 rows of 32 hit distinct banks at any rotation.
__device__ __forceinline__ uint32_t acc_pos(uint32_t m) { return m ^ ((m >> 1) & 16u); }

// Transposition buffer of 16 rows x 32 words: unit u (4 words) of row f at
// u ^ row_rot(f).  The factors' 16-byte stores and the reads of 16 columns x 2
// rows f, f + 8 are free of bank conflicts.
__host__ __device__ constexpr uint32_t row_rot(uint32_t f) { return (f & 3u) ^ (((f >> 3) & 1u) << 2); }

__device__ __forceinline__ uint32_t shoup_k(uint32_t x, uint32_t w, uint32_t wp, uint32_t p) {
    return x * w - __umulhi(x, wp) * p;
}

// (a0, a1) * c + (b0, b1), two FMAs in one instruction
__device__ __forceinline__ void fma_pair(float &r0, float &r1, float a0, float a1, float c, float b0, float b1) {
    asm("{\n\t.reg .b64 a, b, c, r;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%5, %6};\n\tmov.b64 c, {%4, %4};\n\t"
        "fma.rn.f32x2 r, a, c, b;\n\tmov.b64 {%0, %1}, r;\n\t}\n"
        : "=f"(r0), "=f"(r1)
        : "f"(a0), "f"(a1), "f"(c), "f"(b0), "f"(b1));
}

// Digit l of two words as fp16: byte 3 - l of each, less its offset 128.
template <int L>
__device__ __forceinline__ uint32_t digit_pair(uint32_t w0, uint32_t w1) {
    constexpr uint32_t sel = (3 - L) | ((4 + 3 - L) << 8);  // bytes 1 and 3: any, replaced below
    const uint32_t h = (__byte_perm(w0, w1, sel) & 0x00FF00FFu) | 0x64006400u;  // 1024 + 128 + digit
    const __half2 v = __hsub2(*reinterpret_cast<const __half2 *>(&h), __floats2half2_rn(1152.f, 1152.f));
    return *reinterpret_cast<const uint32_t *>(&v);
}

// The words of this lane's eight coefficients (K slots 8 a + i) as the three
// digits' units of the B operand; unit points at digit 0's, 256 bytes a digit.
__device__ __forceinline__ void store_digits(uint4 *unit, const uint32_t (&w)[8]) {
    unit[0] = make_uint4(digit_pair<0>(w[0], w[1]), digit_pair<0>(w[2], w[3]), digit_pair<0>(w[4], w[5]),
                         digit_pair<0>(w[6], w[7]));
    unit[16] = make_uint4(digit_pair<1>(w[0], w[1]), digit_pair<1>(w[2], w[3]), digit_pair<1>(w[4], w[5]),
                          digit_pair<1>(w[6], w[7]));
    unit[32] = make_uint4(digit_pair<2>(w[0], w[1]), digit_pair<2>(w[2], w[3]), digit_pair<2>(w[4], w[5]),
                          digit_pair<2>(w[6], w[7]));
}

// Forward butterfly: X = U + S V, Y = U - S V + 2 p (no reduction).  Both sums
// have three terms: a sum of two may be issued as a multiply-add, and the
// multiply pipe is the bound (81 % busy; 4096 gates at k = 2 216 -> 213 ms).
__device__ __forceinline__ void fwd_bf(uint32_t &U, uint32_t &V, uint32_t w, uint32_t wp, const PrimeK &q) {
    const uint32_t T = shoup_k(V, w, wp, q.p), u = U;
    U = u + T + q.zero;
    V = u - T + q.p2;
}
// Inverse butterfly with the negated twiddle: X = U + V, Y = S (V - U); off
// is a multiple of p that U is below.
__device__ __forceinline__ void inv_bf(uint32_t &U, uint32_t &V, uint32_t w, uint32_t wp, uint32_t off, uint32_t p) {
    const uint32_t u = U, v = V;
    U = u + v;
    V = shoup_k(v - u + off, w, wp, p);
}

// ---------------------------------------------------------------- matrix products
// Instruction descriptor, kind::f16: fp32 accumulator, fp16 A and B, both
// K-major, N = 48, M = 128.
constexpr uint32_t kWarpIdesc = (1u << 4) | ((48u >> 3) << 17) | ((128u >> 4) << 24);

// Shared-memory matrix descriptor: start, leading (K) and stride (row group)
// byte offsets, descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t operand_desc(uint32_t saddr, uint32_t k_stride) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(k_stride >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) |
           (1ull << 46);
}

__device__ __forceinline__ void tmem_st8(uint32_t addr, const uint4 &a, const uint4 &b) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"r"(addr), "r"(a.x),
                 "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}

// Warps 0-3 of a CTA: their rows of the A operand into TMEM.
template <int D>
__device__ __forceinline__ void fill_operands(uint32_t tmem, const uint4 *table, int warp, int lane) {
    using O = Operands<D>;
    const uint32_t at = tmem + ((uint32_t)(32 * warp) << 16);
    const uint4 *row = table + kTabSmall + 32 * warp + lane;
#pragma unroll
    for (int st = 0; st < 2; ++st)
        tmem_st8(at + O::start + 8 * st, __ldg(row + 3 * kTabPlane + 128 * st), make_uint4(0, 0, 0, 0));
#pragma unroll
    for (int b = 4 * O::first; b < 12; ++b)
        tmem_st8(at + O::planes + 8 * (b - 4 * O::first), __ldg(row + 256 * b), __ldg(row + 256 * b + 128));
    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
}

// One thread: the three planes' products of the digits at `digits` (15 MMAs)
// into the 144 TMEM columns at d, then a commit to the mbarrier.  tmem: the
// CTA's columns; ones, plane0: shared-memory addresses.
template <int D>
__device__ __forceinline__ void issue_products(uint32_t tmem, uint32_t d, uint32_t ones, uint32_t plane0,
                                               uint32_t digits, uint32_t bar) {
    using O = Operands<D>;
    const uint64_t bone = operand_desc(ones, kBUnit), bdig = operand_desc(digits, kBUnit);
    const uint64_t aplane = operand_desc(plane0, kAUnit);
#pragma unroll
    for (int pl = 0; pl < 3; ++pl) {
#pragma unroll
        for (int ks = -1; ks < 4; ++ks) {
            const uint64_t bd = ks < 0 ? bone : bdig + ks * (2 * kBUnit / 16);
            const uint32_t acc = ks < 0 ? 0u : 1u;
            if (ks >= 0 && pl < O::first) {
                asm volatile(
                    "{\n\t.reg .pred p;\n\t"
                    "setp.ne.b32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d + 48 * pl),
                    "l"(aplane + ks * (2 * kAUnit / 16)), "l"(bd), "r"(kWarpIdesc), "r"(acc));
            } else {
                const uint32_t at = tmem + (ks < 0 ? O::start + (pl ? 8 : 0) : O::planes + 32 * (pl - O::first) + 8 * ks);
                asm volatile(
                    "{\n\t.reg .pred p;\n\t"
                    "setp.ne.b32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d + 48 * pl),
                    "r"(at), "l"(bd), "r"(kWarpIdesc), "r"(acc));
            }
        }
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// Wait for a gate's products, bounded in global time.  Nothing branches on
// the outcome: a wait that runs out sets the abort and status words (mk_sync
// reports MK_ETIMEOUT), later waits of the CTA return at once, and its gates
// run to their end on whatever TMEM holds: their results are garbage.
__device__ __noinline__ void products_wait(uint32_t bar, uint32_t parity, volatile uint32_t *abort, uint64_t wait_ns,
                                           uint32_t *status) {
    if (*abort) return;
    const uint64_t t0 = st_globaltimer();
    for (uint32_t it = 0; it < (1u << 30); ++it) {
        if (st_mbar_try(bar, parity)) return;
        if (*abort) return;
        if (st_globaltimer() - t0 > wait_ns) break;
    }
    *abort = 1u;
    atomicOr(status, kStatusWarp);
}

// One lane of the warp (the compiler keeps the uniform registers that the
// matrix instructions take their operands from in such a branch: the issue of
// a step's products is on the critical path in the team kernel, one gate 6.75
// -> 6.57 ms; the warp kernel, where it is not, measured slower with it).
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(r));
    return r != 0;
}

// The end of a CTA, by all its threads: waits for every product that its
// threads have issued and gives TMEM back.  After a wait that ran out nothing
// else says that they have completed: later waits return at once, and a barrier
// that missed a commit is a phase behind.  The thread that issued a gate's (a
// team's) products commits them to an mbarrier in the tables' first bytes, which
// are free once all have arrived, and waits with a bound of its own.  ELECT:
// that thread is the first warp's elected lane, else its lane 0.  TMEM_AT: where
// in shared memory the address of the CTA's COLUMNS columns lies.  Not inlined,
// and with one argument: in the kernels' own code the same lines changed the
// register allocation of their loops (4096 gates at k = 2 1.5 to 7 % slower, 96
// at k = 8 1.7 %).
constexpr uint64_t kDrainNs = 1000000000ull;
template <uint32_t COLUMNS, size_t TMEM_AT, bool ELECT>
__device__ __noinline__ void release_tmem(uint32_t *status) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t *tmem = reinterpret_cast<const uint32_t *>(smem + TMEM_AT);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const bool first = ((threadIdx.x >> 5) & 3) == 0;
    if (ELECT ? (first && elect_one()) : (threadIdx.x & 127) == 0) {
        const uint32_t bar = st_smem_addr(smem) + 8 * (threadIdx.x >> 7);
        st_mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        st_fence_proxy_async();
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
        const uint64_t t0 = st_globaltimer();
        bool done = false;
        for (uint32_t it = 0; it < (1u << 30) && !done; ++it) {
            done = st_mbar_try(bar, 0);
            if (!done && st_globaltimer() - t0 > kDrainNs) break;
        }
        if (!done) atomicOr(status, kStatusWarp);
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(*tmem), "r"(COLUMNS) : "memory");
    __syncwarp();
}

__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
          "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
        : "r"(addr));
}

// Sums of the three planes for this thread's factor of one digit polynomial
// (columns tmem, tmem + 48, tmem + 96), and the factor's elements from them,
// below 3.6 p.
struct PlaneSums {
    float f0[16], f1[16], f2[16];
};
__device__ __forceinline__ void fetch_sums(PlaneSums &f, uint32_t tmem) {
    tmem_ld16(tmem, f.f0);
    tmem_ld16(tmem + 48, f.f1);
    tmem_ld16(tmem + 96, f.f2);
}
__device__ __forceinline__ void sums_fetched() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void combine_planes(uint32_t (&x)[16], const PlaneSums &f, const PrimeK &q) {
#pragma unroll
    for (int e = 0; e < 16; e += 2) {
        float g0, g1;
        fma_pair(g0, g1, f.f1[e], f.f1[e + 1], q.c1, q.kf, q.kf);
        fma_pair(g0, g1, f.f2[e], f.f2[e + 1], q.c2, g0, g1);
        x[e] = __float_as_uint(f.f0[e]) + (__float_as_uint(f.f1[e]) << 9) + (__float_as_uint(f.f2[e]) << 18) -
               __float_as_uint(g0) * q.p;
        x[e + 1] = __float_as_uint(f.f0[e + 1]) + (__float_as_uint(f.f1[e + 1]) << 9) +
                   (__float_as_uint(f.f2[e + 1]) << 18) - __float_as_uint(g1) * q.p;
    }
}
__device__ __forceinline__ void load_factor(uint32_t (&x)[16], uint32_t tmem, const PrimeK &q) {
    PlaneSums f;
    fetch_sums(f, tmem);
    sums_fetched();
    combine_planes(x, f, q);
}

// One forward stage at distance 2^LG in the lane's half rows of NP
// polynomials; `heap`: unit u of the lane's twiddles at heap[32 u].
template <int NP, int LG>
__device__ __forceinline__ void half_stage(uint32_t (&x)[NP][16], const uint4 *heap, const PrimeK &q) {
    constexpr int t = 1 << LG, b = 8 >> LG, units = (b + 1) / 2;
#pragma unroll
    for (int u = 0; u < units; ++u) {
        const uint4 S = heap[32 * (b / 2 + u)];
#pragma unroll
        for (int h = (b == 1 ? 1 : 0); h < 2; ++h) {  // entry 0 is unused
            const int i = b == 1 ? 0 : 2 * u + h;
            const uint32_t w = h ? S.z : S.x, wp = h ? S.w : S.y;
#pragma unroll
            for (int a = 0; a < t; ++a)
#pragma unroll
                for (int l = 0; l < NP; ++l) fwd_bf(x[l][2 * t * i + a], x[l][2 * t * i + a + t], w, wp, q);
        }
    }
}

// x below `from` p (a power of two) -> below `to` p.
__device__ __forceinline__ uint32_t reduce_to(uint32_t x, int from, int to, const PrimeK &q) {
    if (from > 8 && to <= 8) x = min(x, x - q.p8);
    if (from > 4 && to <= 4) x = min(x, x - q.p4);
    if (from > 2 && to <= 2) x = min(x, x - q.p2);
    return x;
}

__device__ __forceinline__ uint32_t multiple(int m, const PrimeK &q) { return m == 2 ? q.p2 : (m == 4 ? q.p4 : q.p8); }

// Sums that element c has been through before inverse stage s since its last
// product (or the start); its bound is 2^(1 + sums) p on inputs below 2 p, and
// at 16 p (three sums) it is brought below 2 p before the next stage.
__device__ __forceinline__ int inv_sums(int s, int c) {
    const int low = c & ((1 << s) - 1);
    return low ? s - 1 - (31 - __clz(low)) : s;
}

// Inverse stage s (distance 2^s) in the lane's half row.  The inverse twiddle
// of (b, i) is minus the forward one of (b, b - 1 - i) of half row 63 - y:
// `heap` is that half row's.
template <int s>
__device__ __forceinline__ void half_inverse_stage(uint32_t (&y)[16], const uint4 *heap, const PrimeK &q) {
    constexpr int t = 1 << s, b = 8 >> s, units = (b + 1) / 2;
#pragma unroll
    for (int c = 0; c < 16; ++c)
        if (inv_sums(s, c) == 3) y[c] = reduce_to(y[c], 16, 2, q);
#pragma unroll
    for (int u = 0; u < units; ++u) {
        const uint4 S = heap[32 * (b / 2 + u)];
#pragma unroll
        for (int h = (b == 1 ? 1 : 0); h < 2; ++h) {
            const int i = b == 1 ? 0 : b - 1 - (2 * u + h);
            const uint32_t w = h ? S.z : S.x, wp = h ? S.w : S.y;
#pragma unroll
            for (int a = 0; a < t; ++a) {
                const int c = 2 * t * i + a;  // both operands have been through as many sums
                inv_bf(y[c], y[c + t], w, wp, multiple(2 << (inv_sums(s, c) % 3), q), q.p);
            }
        }
    }
}

// CRT (Garner) of residues x1 mod p1, x2 mod p2, each below 4 p, to the exact
// integer mod 2^32: t p1 + x1 with t = (x2 - x1) / p1 mod p2 taken in
// (-p2/2, p2/2).  x1 need not be canonical (t follows it), and the integers
// are below 2^52.8 in magnitude against p1 p2 / 2 > 2^54.9, so t is never near
// its boundary.  t comes centred from a product that is offset by h =
// (p2 - 1) / 2: the operand is offset by h p1 mod p2.
constexpr uint32_t CRT_H = (P2 - 1) / 2, CRT_HP1 = (uint32_t)((uint64_t)CRT_H * P1 % P2);
__device__ __forceinline__ uint32_t crt_centred(uint32_t x1, uint32_t x2) {
    const uint32_t t = shoup_k(x2 - x1 + (5 * P2 + CRT_HP1), CRT_C, CRT_CP, P2);
    return min(t, t - P2) * P1 + (x1 - CRT_H * P1);
}

// Inverse transform of this lane's half row of residues (below 4 p), and
// recombination: z[i] is the integer (mod 2^32) of coefficient c + 16 (i % 2) +
// 32 (a + 8 (i / 2)), c = lane % 16, a = 2 warp + lane / 16.
//   heap: of half row 63 - y; rows, cross: this prime's tables; crosses: both
//   primes' (prime 1's is 16 units on); ex: the gate's exchange buffer.
__device__ __forceinline__ void inverse_crt(uint32_t (&y)[16], uint32_t (&z)[8], const uint4 *heap, const uint4 *rows,
                                            const uint4 *cross, const uint4 *crosses, uint32_t *xb,
                                            const uint32_t *ex, const PrimeK &q, int h, int warp, int lane, int bar) {
#pragma unroll
    for (int c = 0; c < 16; ++c) y[c] = min(y[c], y[c] - q.p2);
    half_inverse_stage<0>(y, heap, q);
    half_inverse_stage<1>(y, heap, q);
    half_inverse_stage<2>(y, heap, q);
    half_inverse_stage<3>(y, heap, q);
#pragma unroll
    for (int c = 0; c < 16; ++c) {
        const int r = inv_sums(4, c), sums = r > 3 ? r - 3 : r;
        y[c] = reduce_to(y[c], 2 << sums, 4, q);
    }
    {
        uint4 *mine = reinterpret_cast<uint4 *>(xb) + (lane >> 1) * 8;
        const uint32_t first = (4 * (lane & 1)) ^ row_rot(lane >> 1);
#pragma unroll
        for (int u = 0; u < 4; ++u) mine[u ^ first] = make_uint4(y[4 * u], y[4 * u + 1], y[4 * u + 2], y[4 * u + 3]);
    }
    __syncwarp();
    // Lane (rr = lane % 16, fh = lane / 16): columns rr and rr + 16 of rows
    // 16 h + 8 fh + j: d[j] and d[8 + j], below 4 p.
    const uint32_t rr = lane & 15, fh = lane >> 4;
    uint32_t d[16];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t *row = xb + (8 * fh + j) * 32 + (rr & 3);
        const uint32_t u = (rr >> 2) ^ row_rot(j) ^ (4 * fh);
        d[j] = row[4 * u];
        d[8 + j] = row[4 * (u ^ 4)];
    }
    // stage 5: (r, r + 16) with row f's twiddle (minus entry 31 - f of the rows)
    const int base = 31 - 16 * h - 8 * (int)fh;  // odd
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint4 S = rows[(base >> 1) - u];  // entries base - 2u - 1, base - 2u
        inv_bf(d[2 * u], d[8 + 2 * u], S.z, S.w, q.p4, q.p);
        inv_bf(d[2 * u + 1], d[9 + 2 * u], S.x, S.y, q.p4, q.p);
    }
    // d[0..7] below 8 p, d[8..15] below 2 p.  Stages 6 to 8: rows j at distances 1, 2, 4
    const int blk = 2 * h + fh;  // block of 8 rows
#pragma unroll
    for (int u = 0; u < 2; ++u) {  // distance 1: entries 16 + 15 - (4 blk + i)
        const uint4 S = cross[(31 - 4 * blk) / 2 - u];
        inv_bf(d[4 * u], d[4 * u + 1], S.z, S.w, q.p8, q.p);
        inv_bf(d[4 * u + 2], d[4 * u + 3], S.x, S.y, q.p8, q.p);
        inv_bf(d[8 + 4 * u], d[9 + 4 * u], S.z, S.w, q.p2, q.p);
        inv_bf(d[10 + 4 * u], d[11 + 4 * u], S.x, S.y, q.p2, q.p);
    }
#pragma unroll
    for (int j = 0; j < 8; j += 2) d[j] = reduce_to(d[j], 16, 2, q);
    {  // distance 2: entries 8 + 7 - (2 blk + i); d[0..7] below 2 p, d[8 + j] below 4 p (j even) or 2 p
        const uint4 S = cross[(15 - 2 * blk) / 2];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            inv_bf(d[a], d[a + 2], S.z, S.w, q.p2, q.p);
            inv_bf(d[4 + a], d[6 + a], S.x, S.y, q.p2, q.p);
            inv_bf(d[8 + a], d[10 + a], S.z, S.w, a ? q.p2 : q.p4, q.p);
            inv_bf(d[12 + a], d[14 + a], S.x, S.y, a ? q.p2 : q.p4, q.p);
        }
    }
    {  // distance 4: entry 4 + 3 - blk; below 4 p (j < 2) or 2 p, and 8 p, 4 p, 2 p, 2 p
        const uint4 S2 = cross[(7 - blk) / 2];
        const uint32_t w = (blk & 1) ? S2.x : S2.z, wp = (blk & 1) ? S2.y : S2.w;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            inv_bf(d[a], d[a + 4], w, wp, a < 2 ? q.p4 : q.p2, q.p);
            inv_bf(d[8 + a], d[12 + a], w, wp, a == 0 ? q.p8 : (a == 1 ? q.p4 : q.p2), q.p);
        }
    }
    // bounds now: d[0..1] 8 p, d[2..3] 4 p, d[8] 16 p, d[9] 8 p, d[10..11] 4 p, the rest 2 p
    d[0] = reduce_to(d[0], 8, 4, q);
    d[1] = reduce_to(d[1], 8, 4, q);
    d[8] = reduce_to(d[8], 16, 4, q);
    d[9] = reduce_to(d[9], 8, 4, q);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        // row 8 fh + j of this warp's 16 rows of the exchange buffer
        uint32_t *row = xb + (8 * fh + j) * 32;
        const uint32_t c = rr ^ (16 * ((j ^ fh) & 1));  // swapped halves: conflict-free here and below
        row[c] = d[j];
        row[c ^ 16] = d[8 + j];
    }
    quad_sync(bar);
    // Last two stages, both primes: rows a, a + 8, a + 16, a + 24 of columns c and c + 16
    const uint32_t a = 2 * warp + fh;
    uint32_t res[2][8];
#pragma unroll
    for (int pr = 0; pr < 2; ++pr) {
        const uint32_t p = pr ? P2 : P1;
        const uint4 S1 = crosses[16 * pr], S2 = crosses[16 * pr + 1];  // entries 1 (in zw); 2, 3
        const uint32_t *src = ex + pr * 1024 + a * 32 + rr;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            uint32_t v[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) v[b] = src[256 * b + ((g ^ b ^ fh) & 1 ? 16 : 0)];
            inv_bf(v[0], v[1], S2.z, S2.w, 4 * p, p);
            inv_bf(v[2], v[3], S2.x, S2.y, 4 * p, p);
            inv_bf(v[0], v[2], S1.z, S1.w, 8 * p, p);
            inv_bf(v[1], v[3], S1.z, S1.w, 2 * p, p);
            v[0] = min(v[0], v[0] - 8 * p);
            v[0] = min(v[0], v[0] - 4 * p);
#pragma unroll
            for (int b = 0; b < 4; ++b) res[pr][g + 2 * b] = v[b];
        }
    }
    quad_sync(bar);  // every read of the exchange buffer is done
#pragma unroll
    for (int c = 0; c < 8; ++c) z[c] = crt_centred(res[0][c], res[1][c]);
}

// x0 k0 + x1 k1 + x2 k2 (Montgomery keys), below 3.6 p for x below 13.6 p.
__device__ __forceinline__ uint32_t mac3_redc(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t k0, uint32_t k1,
                                              uint32_t k2, const PrimeK &q) {
    uint64_t t = (uint64_t)x0 * k0;
    t += (uint64_t)x1 * k1;
    t += (uint64_t)x2 * k2;
    const uint32_t h = __umulhi((uint32_t)t * q.pinv, q.p);
    return (uint32_t)(t >> 32) - h + q.p;
}

// Units `low` of the lane's factor in three polynomials of each of two keys.
__device__ __forceinline__ void load_keys(uint4 (&key)[6], const uint4 *k1, const uint4 *k2, uint32_t low,
                                          uint32_t eighth) {
    const uint32_t pos = low * 32 + (eighth ^ low);
#pragma unroll
    for (int l = 0; l < 6; ++l) {
        const uint4 *src = (l < 3 ? k1 : k2) + (l % 3) * 512 + pos;
        asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(key[l].x), "=r"(key[l].y), "=r"(key[l].z), "=r"(key[l].w)
                     : "l"(src));
    }
}

// The same units of one key.
__device__ __forceinline__ void load_key(uint4 (&key)[3], const uint4 *k1, uint32_t low, uint32_t eighth) {
    const uint32_t pos = low * 32 + (eighth ^ low);
#pragma unroll
    for (int l = 0; l < 3; ++l)
        asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];\n"
                     : "=r"(key[l].x), "=r"(key[l].y), "=r"(key[l].z), "=r"(key[l].w)
                     : "l"(k1 + l * 512 + pos));
}

__device__ __forceinline__ uint32_t word_of(const uint4 &a, int h) {
    return h == 0 ? a.x : (h == 1 ? a.y : (h == 2 ? a.z : a.w));
}

// HOOK: the instance that withholds a step's products (LaunchShape's
// skip_key_step); the comparison in the loop costs the other one 2.8 % (4096
// gates at k = 2).
template <bool HOOK>
__global__ void __launch_bounds__(128 * kWarpMaxGates, 1)
bootstrap_warp_kernel(LaunchShape S, DeviceKeys K, const GateDesc *__restrict__ desc,
                      const uint32_t *__restrict__ ct_a, const uint32_t *__restrict__ ct_b,
                      const uint32_t *__restrict__ abar_in, int64_t max_steps, uint32_t *__restrict__ ext,
                      uint32_t *__restrict__ acc_out, uint32_t count) {
    constexpr int N = 1024;
    extern __shared__ __align__(16) unsigned char smem[];
    const int k = (int)S.k, n = (int)S.n;
    const uint32_t G = blockDim.x >> 7;
    const WarpLayout L = warp_layout(S.k, S.n, G);
    uint4 *tab = reinterpret_cast<uint4 *>(smem);
    {
        const uint4 *src = static_cast<const uint4 *>(K.tw_warp);
        for (int u = threadIdx.x; u < Operands<kWarpMaxGates>::units; u += blockDim.x) tab[u] = src[u];
    }
    WarpCtl *ctl = reinterpret_cast<WarpCtl *>(smem + L.ctl);
    constexpr uint32_t columns = Operands<kWarpMaxGates>::columns;
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
    st_fence_proxy_async();  // the tables are operands of the matrix products
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    // the warp's index by a shuffle: uniform to the compiler, so constants and bases need no vector registers
    const int wid = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);
    if (wid < 4) fill_operands<kWarpMaxGates>(ctl->tmem, static_cast<const uint4 *>(K.tw_warp), wid, threadIdx.x & 31);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const int lane = threadIdx.x & 31, warp = wid & 3, slot = wid >> 2, t128 = threadIdx.x & 127;
    const int pr = warp >> 1, h = warp & 1, bar = 1 + slot;
    unsigned char *gm = smem + L.gate + L.gate_bytes * slot;
    uint32_t *acc = reinterpret_cast<uint32_t *>(gm + L.acc);
    uint4 *digits = reinterpret_cast<uint4 *>(gm + L.digits);
    uint32_t *ex = reinterpret_cast<uint32_t *>(gm + L.xbuf), *xb = ex + 512 * warp;
    uint4 *park = reinterpret_cast<uint4 *>(gm + L.park) + warp * 128 + lane;
    uint16_t *abar = reinterpret_cast<uint16_t *>(gm + L.abar);
    const uint4 *heap = tab + warp * 256 + lane, *heap_rev = tab + (warp ^ 1) * 256 + 31 - lane;
    const uint4 *rows = tab + kTabHalves + pr * 16;
    const uint4 *crosses = tab + kTabHalves + kTabRows;
    const uint32_t ones_s = st_smem_addr(crosses + kTabCross), plane0_s = ones_s + 16 * kTabOnes;
    const uint32_t digits_s = st_smem_addr(digits);
    const uint32_t mbar = st_smem_addr(&ctl->bar[slot]);
    const uint32_t tmem = ctl->tmem + 144 * slot, tmem_mine = tmem + ((uint32_t)(32 * warp) << 16);
    const PrimeK q = prime_of(pr, S.d - 3);
    const Gadget gad = make_gadget(8);
    const uint4 *bk_all = static_cast<const uint4 *>(K.bk);
    const uint4 *keyA = static_cast<const uint4 *>(K.keyA);
    constexpr int POLY = N / 2;  // 16-byte units of a key polynomial (a plane of 256 per prime)
    const int all_steps = k * n;
    const int limit = (max_steps >= 0 && max_steps < all_steps) ? (int)max_steps : all_steps;
    // this lane's coefficients: c + 16 (i % 2) + 32 (a + 8 (i / 2)), i < 8, c = lane % 16, a = 2 warp + lane / 16;
    // their digits are unit a, column c of each digit
    const uint32_t m0 = (lane & 15) + 32 * (2 * warp + (lane >> 4)), sw0 = acc_pos(m0);
    uint4 *unit = digits + (2 * warp + (lane >> 4)) * (kBUnit / 16) + (lane & 15);
    // its key units: factor y = 32 h + lane, unit v at (u % 8) 32 + (u / 8 xor u % 8), u = 4 y + v
    const uint32_t half_odd = 4 * (lane & 1), eighth = 16 * h + (lane >> 1);
    uint32_t phase = 0;  // products waited for

    for (uint32_t gate = blockIdx.x + gridDim.x * slot; gate < count; gate += gridDim.x * G) {
        if (abar_in) {
            const uint32_t W = S.k * S.n + 1;
            for (uint32_t x = t128; x < W; x += 128) abar[x] = (uint16_t)abar_in[(size_t)gate * W + x];
        } else {
            lin_modswitch(S, desc[gate], ct_a, ct_b, abar, t128, 128);
        }
        quad_sync(bar);
        {
            const uint32_t bbar = abar[k * n];
            for (uint32_t m = t128; m < (uint32_t)N; m += 128) {
                const uint32_t r = (m + bbar) & (2 * N - 1);
                acc[acc_pos(m)] = (r >= (uint32_t)N) ? (0u - (1u << 29)) : (1u << 29);
            }
            for (uint32_t x = N + t128; x < (uint32_t)(k + 1) * N; x += 128) acc[x] = 0;
        }
        quad_sync(bar);
        // The digits of (X^-e - 1) ACC_jj, and one thread's issue of their products once all are stored.
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
        auto start_products = [&](bool issue) {
            st_fence_proxy_async();
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            quad_sync(bar);
            if (warp == 0 && lane == 0 && issue) {
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                issue_products<kWarpMaxGates>(ctl->tmem, tmem, ones_s, plane0_s, digits_s, mbar);
            }
            __syncwarp();
        };
        // Slots 0..k of a step: accumulator polynomials, the other parties' first, then 0, then i;
        // slot k + 1: the digits of v.
        auto poly_of = [k](int s, int i) { return s < k - 1 ? (s + 1 < i ? s + 1 : s + 2) : (s == k - 1 ? 0 : i); };
        auto next_step = [&](int s) {  // e = 0: X^0 - 1 = 0, every digit is 0, the product adds nothing
            while (s < limit && abar[s] == 0) ++s;
            return s;
        };
        bool started = false;  // slot 0's products of this step are under way
        int next = 0;
#pragma unroll 1
        for (int step = next_step(0); step < limit; step = next) {
            const int i = step / n + 1;
            const uint32_t e = abar[step];
            const bool issue = !HOOK || step != S.skip_key_step;
            next = next_step(step + 1);
            const uint4 *bk = bk_all + (size_t)step * 9 * POLY + pr * (POLY / 2);
            uint32_t V[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) V[c] = 0;
            if (!started) {
                cut_digits(poly_of(0, i), e);
                start_products(issue);
            }
            // The next step's first slot can start in this step's last one if its polynomial is final by then:
            // another party's, so not one of this step's 0 and i.
            started = k > 1 && next < limit && next / n + 1 == i;
#pragma unroll 1
            for (int s = 0; s <= k + 1; ++s) {
                const int jj = poly_of(s, i);
                if (!st_mbar_try(mbar, phase & 1)) products_wait(mbar, phase & 1, &ctl->abort, S.wait_ns, K.status);
                ++phase;
                __syncwarp();
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                uint32_t x[3][16];
                load_factor(x[0], tmem_mine, q);
                load_factor(x[1], tmem_mine + 16, q);
                load_factor(x[2], tmem_mine + 32, q);
                // the next slot's products run under this one's butterflies
                if (s < k || (s == k + 1 && started)) {
                    cut_digits(s < k ? poly_of(s + 1, i) : poly_of(0, i), s < k ? e : abar[next]);
                    start_products(s < k ? issue : !HOOK || next != S.skip_key_step);
                }
                // R1 = <x, key1>, R2 = <x, key2> in place of x[0], x[1]: (d, A_jj), or (f0, f1) of v's digits
                const uint4 *k1 = bk + (s <= k ? 0 : 3 * POLY);
                const uint4 *k2 = s <= k ? keyA + (size_t)jj * 3 * POLY + pr * (POLY / 2) : bk + 6 * POLY;
                uint4 key[6];  // the first group is on its way during the butterflies
                load_keys(key, k1, k2, half_odd, eighth);
                half_stage<3, 3>(x, heap, q);
                half_stage<3, 2>(x, heap, q);
                half_stage<3, 1>(x, heap, q);
                half_stage<3, 0>(x, heap, q);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
#pragma unroll
                    for (int e4 = 0; e4 < 4; ++e4) {
                        const int c = 4 * v + e4;
                        const uint32_t x0 = x[0][c], x1 = x[1][c], x2 = x[2][c];
                        x[0][c] = mac3_redc(x0, x1, x2, word_of(key[0], e4), word_of(key[1], e4), word_of(key[2], e4), q);
                        x[1][c] = mac3_redc(x0, x1, x2, word_of(key[3], e4), word_of(key[4], e4), word_of(key[5], e4), q);
                    }
                    if (v < 3) load_keys(key, k1, k2, half_odd + v + 1, eighth);
                }
                // phase A: v += R2, R1 is c'_jj; phase B: c'_0 += R1, c'_i (kept in V) += R2
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const uint32_t a = V[c] + x[1][c];
                    V[c] = min(a, a - q.p4);
                }
                if (s == k - 1) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) park[32 * v] = make_uint4(x[0][4 * v], x[0][4 * v + 1], x[0][4 * v + 2], x[0][4 * v + 3]);
                    continue;
                }
                if (s == k + 1) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const uint4 o = park[32 * v];
#pragma unroll
                        for (int e4 = 0; e4 < 4; ++e4) {
                            const uint32_t a = word_of(o, e4) + x[0][4 * v + e4];
                            x[0][4 * v + e4] = min(a, a - q.p4);
                        }
                    }
                }
                // Inverse transforms due: the others' c'; v; c'_0 and c'_i
                const int jobs = s == k + 1 ? 2 : 1;
#pragma unroll 1
                for (int job = 0; job < jobs; ++job) {
                    uint32_t y[16], z[8];
                    if (s != k) {
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            y[c] = x[0][c];
                            x[0][c] = V[c];  // the second job's
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            y[c] = V[c];
                            V[c] = x[0][c];
                        }
                    }
                    inverse_crt(y, z, heap_rev, rows, crosses + pr * 16, crosses, xb, ex, q, h, warp, lane, bar);
                    if (s == k) {
#pragma unroll
                        for (int c = 0; c < 8; ++c) z[c] += gad.offset;
                        store_digits(unit, z);
                        start_products(issue);
                    } else {
                        uint32_t *ap = acc + (s == k + 1 ? (job ? i : 0) : jj) * N;
#pragma unroll
                        for (int c = 0; c < 8; ++c) ap[(sw0 ^ (16 * (c & 1))) + 256 * (c >> 1)] += z[c];
                    }
                }
            }
            quad_sync(bar);
        }
        if (acc_out) {
            uint32_t *dst = acc_out + (size_t)gate * (k + 1) * N;
            for (uint32_t x = t128; x < (uint32_t)(k + 1) * N; x += 128) dst[x] = acc[(x & ~(N - 1)) + acc_pos(x & (N - 1))];
        } else {
            uint32_t *dst = ext + (size_t)gate * (k * N + 1);
            for (int i = 1; i <= k; ++i)
                for (int m = t128; m < N; m += 128)
                    dst[(i - 1) * N + m] = m == 0 ? acc[i * N] : 0u - acc[i * N + acc_pos(N - m)];
            if (t128 == 0) dst[k * N] = acc[0] + (1u << 29);  // +1/8
        }
        quad_sync(bar);
    }
    constexpr size_t tmem_at = (size_t)Operands<kWarpMaxGates>::units * 16 + offsetof(WarpCtl, tmem);
    release_tmem<columns, tmem_at, false>(K.status);
}

}  // namespace br
}  // namespace mk
