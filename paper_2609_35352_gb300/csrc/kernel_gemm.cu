// kernel_gemm.cu -- the hybrid layer with constant raw plaintexts as exact
// matrix products on the tensor cores (gemm.h has the arithmetic and the
// geometry).
//
// Persistent CTAs walk contiguous ranges of units (limb, 128 coefficients,
// poly; polys fastest, so that gamma's tile comes from L2 the second time).
// Per unit, 16 warps
//   1. read the inputs' residues (each lane one coefficient, coalesced), cut
//      them into digits and write them to tensor memory, in three parts;
//   2. per block of 32 outputs, take the 32 signed sums' accumulators, then
//      those of the two groups of 16 outputs, from tensor memory into
//      registers (which frees the accumulators for the next multiplications,
//      issued by a 17th warp meanwhile), put the digit classes together, add
//      S gamma, reduce once (Sec. 4.2 "Combining the Signed and Raw Routes")
//      and store.
// The digits of G and W are made by the CTA itself when it enters a limb (at
// most twice for a range), from residue 0 of each constant plaintext: no
// workspace, nothing kept between calls.
//
// What bounds it: the epilogue warps' instructions (about 190 an output and 32
// coefficients in all, a third of them integer multiplies; four warps a
// scheduler, half its issue slots used).  Per unit of the 96 -> 96 layer they
// take about 25 k of 32 k cycles, the multiplications (222 of N = 96 or less
// and 108 of N = 32 at the 50 cycles each needs whatever N <= 96) run under
// them but for each unit's first block.  Measured on GB300 (96 -> 96 outputs,
// 4332 constant raw terms, 12 limbs of 2^16): 5.383 ms on the tiled kernel,
// whose products keep the FMA-heavy pipe busy, 1.288 here; the layer's 3.0 GB
// take 0.45 ms.  Each of these made it slower: rolled issue loops (4.3 ms),
// lane-dependent control flow in the issuing warp and 128-bit arithmetic in the
// recombination (2.0), literal digit weights (1.6), the signed sums in registers
// (1.44), the next unit's digits under the last group's epilogue (1.44), 112
// registers a worker by setmaxnreg, the products by gamma formed with the signed
// sums (both 2%).
// All waits are bounded (GemmArgs::wait_ns on the global timer); one that
// gives up sets the context's error flag and the CTA's abort flag, which ends
// every other wait; each warp then stops as a whole, at the end of its unit or
// of a build barrier, and the CTA frees its tensor memory once its
// multiplications in flight have completed.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "async.cuh"
#include "gemm.h"
#include "tc_signed.cuh"

namespace {

typedef unsigned __int128 u128;

constexpr uint32_t kDigits = kGemmDigits, kClasses = kGemmClasses;
constexpr uint32_t kWorkers = kGemmEpilogueWarps * 32;
constexpr uint64_t kDrainNs = 20000000;
constexpr float kMagic = 12582912.0f;          // 1.5 * 2^23
constexpr uint32_t kMagicBits = 0x4B400000u;   // its bits

// sum of 128 2^(8a), a < 5, and 512 2^40: makes the balanced digits of a
// value above -2^49 the bytes (and the upper bits) of an unsigned word
constexpr uint64_t kDigitOffset = 0x8080808080ull + (512ull << 40);

// A pair of fp16 digits: digit J of the offset words a and b (J < 5: byte J
// minus 128; J = 5: bits 40 and up minus 512), by the exact fp16 integers
// 1024 + v
template <int J>
__device__ __forceinline__ uint32_t digit_pair(uint64_t a, uint64_t b)
{
    uint32_t g;
    if constexpr (J < 4) {
        g = __byte_perm((uint32_t)a, (uint32_t)b, J | (J << 4) | ((4 + J) << 8) | ((4 + J) << 12));
    } else if constexpr (J == 4) {
        g = __byte_perm((uint32_t)(a >> 32), (uint32_t)(b >> 32), 0x4400);
    } else {
        g = __byte_perm((uint32_t)(a >> 32), (uint32_t)(b >> 32), 0x6521);
    }
    uint32_t h;
    if constexpr (J < 5)
        h = __byte_perm(g, 0x64646464u, 0x4240);  // 0x6400 | byte in each half
    else
        h = g + 0x64006400u;  // at most 1024 + 1024 (fp16 2048)
    const uint32_t off = J < 5 ? 0x64806480u : 0x66006600u;  // 1152, 1536
    __half2 r = __hsub2(*reinterpret_cast<__half2 *>(&h), *reinterpret_cast<const __half2 *>(&off));
    return *reinterpret_cast<uint32_t *>(&r);
}

template <int J>
__device__ __forceinline__ void store_digit(uint32_t taddr, const uint64_t (&u)[8])
{
    uint32_t v[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = digit_pair<J>(u[2 * m], u[2 * m + 1]);
    tcs::st4(taddr, v);
}

// The multiplications of a block's signed sums (32 columns per input digit)
// and of a group's raw sums, for STEPS steps of 16 inputs; `b` = shared
// address of W or of the group's digits.  Unrolled: with the loops left, the
// one issuing thread took about 370 cycles a multiplication instead of the 50
// the tensor cores need.
template <uint32_t STEPS>
__device__ __forceinline__ void issue_signed_n(uint32_t tmem, uint32_t d0, uint32_t b)
{
    const uint64_t desc = tcs::smem_desc(b, 128, STEPS * 256);
#pragma unroll
    for (uint32_t d = 0; d < kDigits; ++d)
#pragma unroll
        for (uint32_t k = 0; k < STEPS; ++k)
            tcs::mma(tmem + d0 + d * kGemmBlock, tmem + 8 * (d * STEPS + k), desc + 16 * k,
                     tcs::idesc_f16(128, kGemmBlock), k > 0);
}

// The same for part `j`, 32 inputs (the last may have 16), of a unit's first
// block: its digits come in that order.
template <uint32_t STEPS>
__device__ __forceinline__ void issue_signed_part(uint32_t tmem, uint32_t d0, uint32_t b, uint32_t j)
{
    const uint64_t desc = tcs::smem_desc(b, 128, STEPS * 256) + 32 * j;
    const uint32_t dig = tmem + 16 * j;
#pragma unroll
    for (uint32_t d = 0; d < kDigits; ++d)
        tcs::mma(tmem + d0 + d * kGemmBlock, dig + 8 * (d * STEPS), desc, tcs::idesc_f16(128, kGemmBlock), j > 0);
    if (STEPS % 2 && j == STEPS / 2) return;
#pragma unroll
    for (uint32_t d = 0; d < kDigits; ++d)
        tcs::mma(tmem + d0 + d * kGemmBlock, dig + 8 * (d * STEPS + 1), desc + 16, tcs::idesc_f16(128, kGemmBlock), 1);
}

// (A multiplication's columns all accumulate or are all overwritten: digit 0
// of the inputs first writes the classes 0 to 5, and the first 16 inputs of
// digit 5, cut in two, the classes 6 to 10.)
template <uint32_t STEPS>
__device__ __forceinline__ void issue_raw_n(uint32_t tmem, uint32_t d0, uint32_t b)
{
    const uint64_t desc = tcs::smem_desc(b, 128, STEPS * 256);
    constexpr uint32_t id = tcs::idesc_f16(128, 16 * kDigits);
#pragma unroll
    for (uint32_t n = 0; n < kDigits; ++n) {
        const uint32_t d = n == 0 ? 0 : n == 1 ? kDigits - 1 : n - 1;  // 0, 5, 1, 2, 3, 4
        const uint32_t acc = tmem + d0 + d * 16;
#pragma unroll
        for (uint32_t k = 0; k < STEPS; ++k) {
            const uint32_t dig = tmem + 8 * (d * STEPS + k);
            if (n == 1 && k == 0) {
                tcs::mma(acc + 16, dig, desc + STEPS * 32, tcs::idesc_f16(128, 16 * (kDigits - 1)), 0);
                tcs::mma(acc, dig, desc, tcs::idesc_f16(128, 16), 1);
            } else {
                tcs::mma(acc, dig, desc + 16 * k, id, n > 0 || k > 0);
            }
        }
    }
}

#define GEMM_STEPS(F, ...)                              \
    switch (steps) {                                    \
        case 1: F<1>(__VA_ARGS__); break;               \
        case 2: F<2>(__VA_ARGS__); break;               \
        case 3: F<3>(__VA_ARGS__); break;               \
        case 4: F<4>(__VA_ARGS__); break;               \
        case 5: F<5>(__VA_ARGS__); break;               \
        default: F<6>(__VA_ARGS__); break;              \
    }
__device__ __forceinline__ void issue_signed(uint32_t steps, uint32_t tmem, uint32_t d0, uint32_t b)
{
    GEMM_STEPS(issue_signed_n, tmem, d0, b)
}
__device__ __forceinline__ void issue_signed(uint32_t steps, uint32_t tmem, uint32_t d0, uint32_t b, uint32_t j)
{
    GEMM_STEPS(issue_signed_part, tmem, d0, b, j)
}
__device__ __forceinline__ void issue_raw(uint32_t steps, uint32_t tmem, uint32_t d0, uint32_t b)
{
    GEMM_STEPS(issue_raw_n, tmem, d0, b)
}
#undef GEMM_STEPS

// true in one lane of the (converged) warp
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t c)
{
    uint64_t r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ int64_t mad_wide_s(int32_t a, int32_t b, int64_t c)
{
    int64_t r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
// the bits of a small integer plus kMagic
__device__ __forceinline__ uint32_t magic(uint32_t f) { return __float_as_uint(__fadd_rn(__uint_as_float(f), kMagic)); }
__device__ __forceinline__ int32_t to_int(uint32_t f) { return __float2int_rn(__uint_as_float(f)); }

// sum of kMagicBits 2^(8s) for s < n
__host__ __device__ constexpr uint64_t magic_sum(int n)
{
    uint64_t r = 0;
    for (int s = 0; s < n; ++s) r += (uint64_t)kMagicBits << (8 * s);
    return r;
}

// Per output: the bias of the raw sum, cut into the parts of weights 1, 2^32
// and 2^64.  With theirs the words of weights 1 and 2^32 are not negative; b2,
// and the word of weight 2^64 with it, is negative for narrow moduli (t is about
// 2^74 at 34 bits, less 2^18 borrowed here): that word counts modulo 2^64, and the
// sum of the three modulo 2^128, where it is the true one, in [0, 2^(2k+9)).
struct __align__(16) OutBias {
    uint64_t b0, b1, b2, pad;
};

// (l0 + l1 2^32 + l2 2^64 + s g) mod q; the value is below 2^(2k+9) for a
// k-bit q, 34 <= k <= 50, `shift` = k - 34, mk = floor(2^(k+62) / q)
// (written out in words: 128-bit arithmetic in C took about half as many
// instructions again)
__device__ __forceinline__ uint64_t finish(uint64_t l0, uint64_t l1, uint64_t l2, uint64_t s, uint64_t g, uint64_t q,
                                           uint64_t mk, uint32_t shift)
{
    const uint32_t s0 = (uint32_t)s, s1 = (uint32_t)(s >> 32), g0 = (uint32_t)g, g1 = (uint32_t)(g >> 32);
    uint32_t w0 = (uint32_t)l0, w1 = (uint32_t)(l0 >> 32), w2 = (uint32_t)(l1 >> 32), w3 = (uint32_t)(l2 >> 32);
    asm("add.cc.u32 %0, %0, %3;\n\t"
        "addc.cc.u32 %1, %1, %4;\n\t"
        "addc.u32 %2, %2, 0;"
        : "+r"(w1), "+r"(w2), "+r"(w3)
        : "r"((uint32_t)l1), "r"((uint32_t)l2));
    asm("mad.lo.cc.u32 %0, %4, %6, %0;\n\t"
        "madc.hi.cc.u32 %1, %4, %6, %1;\n\t"
        "madc.lo.cc.u32 %2, %5, %7, %2;\n\t"
        "madc.hi.u32 %3, %5, %7, %3;"
        : "+r"(w0), "+r"(w1), "+r"(w2), "+r"(w3)
        : "r"(s0), "r"(s1), "r"(g0), "r"(g1));
    // s < 2^58, g < 2^50: the middle products fit together in 64 bits
    const uint64_t mid = mad_wide(s1, g0, mad_wide(s0, g1, 0));
    asm("add.cc.u32 %0, %0, %3;\n\t"
        "addc.cc.u32 %1, %1, %4;\n\t"
        "addc.u32 %2, %2, 0;"
        : "+r"(w1), "+r"(w2), "+r"(w3)
        : "r"((uint32_t)mid), "r"((uint32_t)(mid >> 32)));
    // quotient: A = floor(x / 2^(k-2)), below 2^61, times mk = floor(2^(k+62) /
    // q), below 2^63, the product's upper half without its lowest partial
    // product: at most 3 below x / q, so the remainder is below 4q
    const uint32_t a0 = __funnelshift_r(w1, w2, shift), a1 = __funnelshift_r(w2, w3, shift);
    const uint32_t m0 = (uint32_t)mk, m1 = (uint32_t)(mk >> 32);
    const uint64_t h = mad_wide(a1, m1, 0) + (mad_wide(a0, m1, mad_wide(a1, m0, 0)) >> 32);
    const uint64_t x0 = ((uint64_t)w1 << 32) | w0;
    const uint64_t r = x0 - h * q;
    const int64_t r1 = (int64_t)(r - 2 * q);
    const uint64_t r2 = r1 < 0 ? r : (uint64_t)r1;
    const int64_t r3 = (int64_t)(r2 - q);
    return r3 < 0 ? r2 : (uint64_t)r3;
}

// what the middle word borrows from the upper one to stay positive (its
// classes sum to less than 2^48.1)
constexpr uint64_t kSplitB1 = 1ull << 50;

// x mod q, x < 2^64
__device__ __forceinline__ uint64_t mod64(uint64_t x, const LimbConst &m) { return rns::reduce64(x, m); }

// A wait whose first try found the phase incomplete.  Giving up (or finding
// that another thread did) leaves `*abort` set; the caller goes on either way and
// looks at the flag where its whole warp can leave.  Out of line: inline, the
// clock and the loops took the 96 -> 96 layer from 1.278 to 1.347 ms.
__device__ __noinline__ void slow_wait(uint32_t bar, uint32_t parity, int *abort, uint64_t limit_ns, int *err)
{
    volatile int *flag = abort;
    if (*flag || async::mbar_wait_bounded(bar, parity, flag, limit_ns) || *flag) return;
    *flag = 1;
    atomicOr(err, 1);
}

__global__ void __launch_bounds__(kGemmThreads, 1) gemm_kernel(const GemmArgs a)
{
    extern __shared__ __align__(128) char sm[];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const GemmLayout lay(a.K, a.chunk);
    const uint32_t tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t base = async::smem_addr(sm);
    const uint32_t bar_full = base + lay.bars, bar_empty = bar_full + 8, bar_build = bar_full + 16;
    const uint32_t bar_drain = bar_full + 48;
    const uint32_t bar_a = bar_full + 24;  // + 8 * part of 32 inputs
    const uint32_t d0 = kDigits * (a.K / 2);  // first accumulator column
    const uint32_t per_limb = a.N / kGemmRows * 2;
    const uint32_t u_begin = (uint32_t)((uint64_t)a.units * blockIdx.x / gridDim.x);
    const uint32_t u_end = (uint32_t)((uint64_t)a.units * (blockIdx.x + 1) / gridDim.x);
    // the first unit's chunk, limb, and place in the limb (2 tile + poly); the
    // walk counts on from there
    struct Unit {
        uint32_t c, l, at;
    };
    const uint32_t first_limb = u_begin / per_limb;
    Unit un{first_limb / a.n_limbs, first_limb % a.n_limbs, u_begin % per_limb};
    auto step = [&](Unit v) {
        if (++v.at == per_limb) {
            v.at = 0;
            if (++v.l == a.n_limbs) {
                v.l = 0;
                ++v.c;
            }
        }
        return v;
    };

    if (tid == 0) {
        s_abort = 0;
        for (uint32_t j = 0; j < kGemmMaxInputs / 32; ++j)
            async::mbar_init(bar_a + 8 * j, kGemmEpilogueWarps + ((a.test_flags & kGemmTestDigits) != 0));
        async::mbar_init(bar_full, 1 + ((a.test_flags & kGemmTestFull) != 0));
        async::mbar_init(bar_drain, 1);
        async::mbar_init(bar_empty, kGemmEpilogueWarps);
        async::mbar_init(bar_build, kGemmEpilogueWarps);
        async::mbar_init_fence();
    }
    if (warp == kGemmEpilogueWarps) tcs::tmem_alloc(async::smem_addr(&s_tmem), 512);
    tcs::fence_before();
    __syncthreads();
    tcs::fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);

    // Waits.  Each lane has its own clock and its own look at the abort flag, and
    // one that left alone would leave the others at a warp-wide instruction: so
    // no wait leaves a loop.  After one that gave up a warp goes on with whatever
    // the operands hold (no address depends on them) and leaves by a vote, at the
    // end of the unit or of a build barrier, which s_gamma's entries depend on.
    auto pass = [&](uint32_t bar, uint32_t parity) {  // (a __syncwarp follows)
        if (!async::mbar_try_wait(bar, parity)) slow_wait(bar, parity, &s_abort, a.wait_ns, a.err);
    };
    auto pass_warp = [&](uint32_t bar, uint32_t parity) {
        if (!__all_sync(0xffffffffu, async::mbar_try_wait(bar, parity)))
            slow_wait(bar, parity, &s_abort, a.wait_ns, a.err);
        __syncwarp();
    };
    auto going = [&] { return __all_sync(0xffffffffu, *(volatile int *)&s_abort == 0) != 0; };
    // one arrival per warp
    auto arrive = [&](uint32_t bar) {
        __syncwarp();
        if (lane == 0) async::mbar_arrive(bar);
    };
    // outputs of a chunk
    auto chunk_outs = [&](uint32_t c) { return min(a.chunk, a.n_out - c * a.chunk); };

    if (warp == kGemmEpilogueWarps) {
        // ---- the multiplications: the whole warp walks the groups (uniform
        // control flow keeps the descriptors in uniform registers), one
        // elected lane issues
        uint32_t n_full = 0, n_unit = 0;
        const uint32_t steps = a.K / 16;
        bool ok = true;
        for (uint32_t u = u_begin; u < u_end && ok; ++u, ++n_unit, un = step(un)) {
            const uint32_t n_out = chunk_outs(un.c);
            for (uint32_t o = 0; o < n_out; o += kGemmBlock) {
                const uint32_t blk = base + (o / kGemmBlock) * lay.block;
                const uint32_t n_groups = n_out - o > 16 ? 2 : 1;
                for (uint32_t g = 0; g <= n_groups; ++g, ++n_full) {
                    if (n_full) pass(bar_empty, (n_full - 1) & 1);
                    tcs::fence_after();
                    __syncwarp();
                    if (o == 0 && g == 0) {
                        for (uint32_t j = 0; j < (steps + 1) / 2; ++j) {
                            pass(bar_a + 8 * j, n_unit & 1);
                            tcs::fence_after();
                            __syncwarp();
                            if (elect_one()) issue_signed(steps, tmem, d0, blk + 2 * lay.group, j);
                            __syncwarp();
                        }
                        if (elect_one()) tcs::commit(bar_full);
                    } else if (elect_one()) {
                        if (g == 0)
                            issue_signed(steps, tmem, d0, blk + 2 * lay.group);
                        else
                            issue_raw(steps, tmem, d0, blk + (g - 1) * lay.group);
                        tcs::commit(bar_full);
                    }
                    __syncwarp();
                }
            }
            ok = going();
        }
        // every multiplication issued completes before the tensor memory goes,
        // whoever gave up
        const int never = 0;
        if (elect_one()) tcs::commit(bar_drain);
        __syncwarp();
        async::mbar_wait_bounded(bar_drain, 0, &never, kDrainNs);
        __syncwarp();
    } else {
        // ---- digits, epilogue
        const uint32_t q4 = warp & 3, k4 = warp >> 2;  // tensor memory quarter; share of the inputs and outputs
        const uint32_t tq = tmem + ((32u * q4) << 16);
        OutBias *bias = reinterpret_cast<OutBias *>(sm + lay.bias);
        uint64_t *s_bias = reinterpret_cast<uint64_t *>(sm + lay.sbias);
        int *wsum = reinterpret_cast<int *>(sm + lay.wsum);
        uint64_t *S = reinterpret_cast<uint64_t *>(sm + lay.sums) + tid;
        unsigned long long *rowsum = reinterpret_cast<unsigned long long *>(sm + lay.rowsum);
        uint32_t *s_gamma = reinterpret_cast<uint32_t *>(sm + lay.gamma);
        uint32_t n_full = 0, n_build = 0;
        uint32_t cur_limb = 0xffffffffu, cur_chunk = 0xffffffffu;
        LimbConst m{};
        uint64_t q = 0, mk = 0;
        uint32_t shift = 0;
        bool ok = true;
        const size_t LN = (size_t)a.L * a.N;
        const uint32_t stride = a.L * a.N * 8;  // bytes between polys (at most 2^26)
        auto build_barrier = [&] {
            arrive(bar_build);
            pass_warp(bar_build, n_build++ & 1);
            return going();
        };
        for (uint32_t u = u_begin; u < u_end && ok; ++u) {
            const Unit v = un;
            un = step(un);
            const uint32_t c = v.c, l = a.limb0 + v.l, poly = v.at & 1, k0 = (v.at >> 1) * kGemmRows;
            const uint32_t n_out = chunk_outs(c), out0 = c * a.chunk;
            // the digits of G and W, and the biases, on entering a limb or chunk
            if (l != cur_limb || c != cur_chunk) {
                if (!(ok = build_barrier())) break;  // every thread is done with the old ones
                m = a.limbs[l];
                q = m.q;
                // floor(2^(k+63) / q) halved is floor(2^(k+62) / q)
                mk = m.mk / 2;
                shift = (uint32_t)m.km1 - 33;
                const uint64_t half = m.q / 2;
                if (c != cur_chunk) {
                    for (uint32_t i = tid; i < lay.bias / 16; i += kWorkers)
                        reinterpret_cast<uint4 *>(sm)[i] = make_uint4(0, 0, 0, 0);
                    for (uint32_t i = tid; i < a.chunk; i += kWorkers) {
                        wsum[i] = 0;
                        s_gamma[i] = i < n_out ? a.gamma[out0 + i] : kGemmNoGamma;
                    }
                }
                for (uint32_t i = tid; i < a.chunk; i += kWorkers) rowsum[i] = 0;
                if (!(ok = build_barrier())) break;
                auto at = [&](uint32_t row, uint32_t col) {  // K-major core matrices of 8 rows x 16 bytes
                    return (row / 8) * (a.K / 8) * 128 + (col / 8) * 128 + (row % 8) * 16 + (col % 8) * 2;
                };
                if (c != cur_chunk)
                    for (uint32_t i = a.sgn_off[c] + tid; i < a.sgn_off[c + 1]; i += kWorkers) {
                        const GemmTerm t = a.sgn[i];
                        char *w = sm + (t.out / kGemmBlock) * lay.block + 2 * lay.group;
                        *reinterpret_cast<__half *>(w + at(t.out % kGemmBlock, t.in)) = __int2half_rn(t.pt ? 1 : -1);
                        atomicAdd(&wsum[t.out], t.pt ? 1 : -1);
                    }
                for (uint32_t i = a.raw_off[c] + tid; i < a.raw_off[c + 1]; i += kWorkers) {
                    const GemmTerm t = a.raw[i];
                    const uint64_t v = a.pt[(size_t)t.pt * LN + (size_t)l * a.N];
                    const int64_t g = v > half ? (int64_t)v - (int64_t)m.q : (int64_t)v;  // centred
                    atomicAdd(&rowsum[t.out], (unsigned long long)g);
                    uint64_t w = (uint64_t)g + kDigitOffset;
                    char *b = sm + (t.out / kGemmBlock) * lay.block + ((t.out / 16) & 1) * lay.group;
#pragma unroll
                    for (uint32_t d = 0; d < kDigits; ++d, w >>= 8) {
                        const int dv = d < 5 ? (int)(w & 255) - 128 : (int)w - 512;
                        *reinterpret_cast<__half *>(b + at(d * 16 + t.out % 16, t.in)) = __int2half_rn(dv);
                    }
                }
                async::fence_proxy_async();
                if (!(ok = build_barrier())) break;
                // sum G (x - half) + half sum G = sum G x, made positive by a
                // multiple of q: |sum G (x - half)| < 96 * 2^(2k - 2), and
                // |sum W (x - half)| < 96 * 2^(k - 1), k the bits of q; less
                // what the magic addends bring
                if (tid < n_out) {
                    const int64_t rs = (int64_t)rowsum[tid];  // |rs| <= 64 * 2^49
                    const uint64_t rq = rs >= 0 ? mod64((uint64_t)rs, m) : m.q - mod64((uint64_t)-rs, m);
                    const uint32_t k = (uint32_t)m.km1 + 1;
                    uint64_t plo, phi;
                    rns::mul_wide(plo, phi, half, rq);
                    const uint64_t corr = rns::reduce128(plo, phi, m);
                    // (q 2^(k+6) >= 2^(2k+5))
                    const u128 t = (u128)m.q * ((uint64_t)1 << (k + 6)) + corr - magic_sum(4);
                    const int ws = wsum[tid];
                    const uint64_t sc = mod64((uint64_t)(ws < 0 ? -ws : ws) * half, m);  // below 96 * 2^49
                    const uint64_t s = (ws < 0 ? m.q - sc : sc) + 128 * m.q;
                    // t = b0 + b1 2^32 + b2 2^64 with b1 >= 2^50 (|l1| < 2^49.1)
                    OutBias b;
                    b.b0 = (uint32_t)t;
                    b.b1 = (uint32_t)((uint64_t)t >> 32) + kSplitB1;
                    b.b2 = (uint64_t)(t >> 64) - (kSplitB1 >> 32);
                    bias[tid] = b;
                    // the signed sum's two words carry kMagicBits in each of six digits
                    s_bias[tid] = s - magic_sum(4) - (magic_sum(2) << 32);
                }
                if (!(ok = build_barrier())) break;
                cur_limb = l;
                cur_chunk = c;
            }

            // 1. the digits of the inputs into tensor memory: this lane's
            //    coefficient, every fourth group of 8 inputs
            {
                const char *x = reinterpret_cast<const char *>(a.in + (size_t)poly * LN + (size_t)l * a.N + k0 + 32 * q4 + lane);
                const uint64_t half = q / 2, off = kDigitOffset - half;
                uint64_t w[kGemmMaxInputs / 32][8];  // every load first
#pragma unroll
                for (uint32_t j = 0; j < kGemmMaxInputs / 32; ++j)
#pragma unroll
                    for (uint32_t i = 0; i < 8; ++i) {
                        const uint32_t in = 8 * (k4 + 4 * j) + i;
                        w[j][i] = in < a.n_in ? __ldg(reinterpret_cast<const uint64_t *>(x + (uint64_t)in * (2 * stride)))
                                              : half;  // (the digits of 0)
                    }
#pragma unroll
                for (uint32_t j = 0; j < kGemmMaxInputs / 32; ++j) {
                    const uint32_t g = k4 + 4 * j;
                    if (g < a.K / 8) {
#pragma unroll
                        for (uint32_t i = 0; i < 8; ++i) w[j][i] += off;
                        const uint32_t t = tq + 4 * g;
                        store_digit<0>(t, w[j]);
                        store_digit<1>(t + (a.K / 2), w[j]);
                        store_digit<2>(t + 2 * (a.K / 2), w[j]);
                        store_digit<3>(t + 3 * (a.K / 2), w[j]);
                        store_digit<4>(t + 4 * (a.K / 2), w[j]);
                        store_digit<5>(t + 5 * (a.K / 2), w[j]);
                    }
                    if (j < (a.K + 31) / 32) {
                        tcs::wait_st();
                        tcs::fence_before();
                        arrive(bar_a + 8 * j);
                    }
                }
            }
            // the next unit's inputs towards L2, and a new tile's gammas
            if (u + 1 < u_end) {
                const size_t at = (size_t)(a.limb0 + un.l) * a.N + (un.at >> 1) * kGemmRows;
                const uint64_t *x = a.in + (size_t)(un.at & 1) * LN + at;
                for (uint32_t i = tid; i < a.n_in * (kGemmRows / 16); i += kWorkers)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(x + (size_t)(i / (kGemmRows / 16)) * 2 * LN +
                                                                 (i % (kGemmRows / 16)) * 16));
                if ((un.at & 1) == 0)
                    for (uint32_t i = tid; i < n_out * (kGemmRows / 16); i += kWorkers) {
                        const uint32_t gj = s_gamma[i / (kGemmRows / 16)];
                        if (gj != kGemmNoGamma)
                            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.pt + (size_t)gj * LN + at +
                                                                         (i % (kGemmRows / 16)) * 16));
                    }
            }

            // 2. the blocks of outputs
            const char *gam = reinterpret_cast<const char *>(a.pt + (size_t)l * a.N + k0 + 32 * q4 + lane);
            char *y = reinterpret_cast<char *>(a.out + ((size_t)(out0 * 2 + poly) * a.L + l) * a.N + k0 + 32 * q4 + lane);
            for (uint32_t o = 0; o < n_out; o += kGemmBlock) {
                const uint32_t n_groups = n_out - o > 16 ? 2 : 1;
                pass_warp(bar_full, n_full++ & 1);
                tcs::fence_after();
                {
                    uint32_t e[2][kDigits][4];
#pragma unroll
                    for (uint32_t d = 0; d < kDigits; ++d) {
                        tcs::ld4(tq + d0 + d * kGemmBlock + 4 * k4, e[0][d]);
                        tcs::ld4(tq + d0 + d * kGemmBlock + 16 + 4 * k4, e[1][d]);
                    }
                    tcs::wait_ld();
                    tcs::fence_before();
                    arrive(bar_empty);
#pragma unroll
                    for (uint32_t g = 0; g < 2; ++g)
#pragma unroll
                        for (uint32_t i = 0; i < 4; ++i) {
                            uint64_t lo = magic(e[g][0][i]), hi = magic(e[g][4][i]);
                            lo = mad_wide(magic(e[g][1][i]), a.c8, lo);
                            lo = mad_wide(magic(e[g][2][i]), a.c16, lo);
                            lo = mad_wide(magic(e[g][3][i]), a.c24, lo);
                            hi = mad_wide(magic(e[g][5][i]), a.c8, hi);
                            // (mod 2^64; the sum is below 2^58)
                            // (kept in shared memory, a slot per thread: the
                            // sixteen registers are needed below)
                            S[(4 * g + i) * kWorkers] = lo + (hi << 32) + s_bias[min(o + 16 * g + 4 * k4 + i, n_out - 1)];
                        }
                }
                // (not unrolled: the group's sums alone take 44 registers)
#pragma unroll 1
                for (uint32_t g = 0; g < n_groups; ++g) {
                    const uint32_t o1 = o + 16 * g + 4 * k4;  // this warp's four outputs
                    uint64_t gm[4];
                    const uint4 g4 = *reinterpret_cast<const uint4 *>(s_gamma + o1);
                    const uint32_t gi[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
                    for (uint32_t i = 0; i < 4; ++i)
                        gm[i] = gi[i] != kGemmNoGamma
                                    ? __ldg(reinterpret_cast<const uint64_t *>(gam + (uint64_t)gi[i] * stride))
                                    : 0;
                    pass_warp(bar_full, n_full++ & 1);
                    tcs::fence_after();
                    char *yo = y + (uint64_t)(o1 * 2) * stride;
                    uint32_t e[kClasses][4];
#pragma unroll
                    for (uint32_t s = 0; s < kClasses; ++s) tcs::ld4(tq + d0 + s * 16 + 4 * k4, e[s]);
                    tcs::wait_ld();
                    tcs::fence_before();
                    arrive(bar_empty);
#pragma unroll
                    for (uint32_t i = 0; i < 4; ++i) {
                        const OutBias b = bias[o1 + i];
                        // the classes as three words of weights 1, 2^32, 2^64,
                        // each with its part of the bias (OutBias)
                        uint64_t l0 = b.b0 + magic(e[0][i]);
                        l0 = mad_wide(magic(e[1][i]), a.c8, l0);
                        l0 = mad_wide(magic(e[2][i]), a.c16, l0);
                        l0 = mad_wide(magic(e[3][i]), a.c24, l0);
                        int64_t l1 = mad_wide_s(to_int(e[4][i]), a.c1, (int64_t)b.b1);
                        l1 = mad_wide_s(to_int(e[5][i]), a.c8, l1);
                        l1 = mad_wide_s(to_int(e[6][i]), a.c16, l1);
                        l1 = mad_wide_s(to_int(e[7][i]), a.c24, l1);
                        int64_t l2 = mad_wide_s(to_int(e[8][i]), a.c1, (int64_t)b.b2);
                        l2 = mad_wide_s(to_int(e[9][i]), a.c8, l2);
                        l2 = mad_wide_s(to_int(e[10][i]), a.c16, l2);
                        const uint64_t v =
                            finish(l0, (uint64_t)l1, (uint64_t)l2, S[(4 * g + i) * kWorkers], gm[i], q, mk, shift);
                        if (o1 + i < n_out) *reinterpret_cast<uint64_t *>(yo) = v;
                        yo += 2 * (size_t)stride;
                    }
                }
            }
            ok = going();
        }
    }
    tcs::fence_before();
    __syncthreads();
    tcs::fence_after();
    if (warp == kGemmEpilogueWarps) {
        __syncwarp();
        tcs::tmem_dealloc(tmem, 512);
    }
}

}  // namespace

int gemm_configure(size_t smem)
{
    return allow_shared_memory((const void *)gemm_kernel, smem, "matrix kernel attribute");
}

uint32_t gemm_units(const fiona_plan *p, uint32_t n_limbs)
{
    const GemmSchedule *g = p->gemm;
    return g->args.n_chunks * n_limbs * (p->ctx->N / kGemmRows) * 2;
}

int launch_gemm(const fiona_plan *p, void *stream, const uint64_t *in, const uint64_t *pt, uint64_t *out, uint32_t l0,
                uint32_t l1, uint32_t layout_L)
{
    const GemmSchedule *g = p->gemm;
    if (l1 <= l0) return FIONA_OK;
    GemmArgs a = g->args;
    a.in = in;
    a.pt = pt;
    a.out = out;
    a.limb0 = l0;
    a.n_limbs = l1 - l0;
    a.L = layout_L;
    a.units = gemm_units(p, a.n_limbs);
    const uint32_t grid = std::min(a.units, (uint32_t)std::max(p->ctx->sm_count, 1));
    gemm_kernel<<<grid, kGemmThreads, g->smem, (cudaStream_t)stream>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(FIONA_ERR_CUDA, "matrix kernel launch: %s", cudaGetErrorString(e));
    return FIONA_OK;
}
