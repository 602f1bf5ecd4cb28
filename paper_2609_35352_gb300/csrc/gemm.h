// gemm.h -- schedule of the matrix kernel for layers with constant raw
// plaintexts (kernel_gemm.cu; built by lower_gemm.cpp).
//
// Column packing (Sec. 6 "BERT") multiplies a ciphertext by one weight in
// every slot, whose plaintext is one residue per limb.  The raw route of such
// a layer is then, limb by limb, a product of the residue matrix G (outputs x
// inputs) with the inputs, the same G for every coefficient of both polys, and
// the signed route's sums are a product with the ternary matrix W: both run
// exactly on the tensor cores, and only the products by gamma (a full
// plaintext per scale group) stay element-wise.
//
// Exactness.  Residues x (and entries g of G, centred to [-q/2, q/2]) of
// 2^33 < q < 2^50 are cut into six balanced digits of radix 2^8, x - floor(q/2) =
// sum_a d_a 2^(8a), |d_a| <= 128 for a < 5 and |d_5| <= 512: integers that
// fp16 holds.  The products of digits a and b with a + b = s add into one
// f32 accumulator, exact while every partial sum is an integer of magnitude
// at most 2^24; with R raw terms in an output the largest class, s = 10, has
// R 2^18, so R <= 64 (kGemmMaxRaw).  (Seven digits of 8 bits take 49 digit
// products and 13 accumulators instead of 36 and 11; digits of 9 bits leave R
// <= 42.)  Classes 0 to 3 stay within R 2^16 <= 2^22, which the epilogue's
// conversion by a magic addend needs, and so do the signed sums' digits
// (96 * 512).
//
// Geometry.  A CTA takes 128 coefficients of one poly and limb (the rows, M =
// 128) and a chunk of the outputs in blocks of 32.  The inputs' digits sit in
// tensor memory (the A operand: K/2 columns per digit, K = inputs rounded up
// to 16), the digits of the CTA's part of G and W in shared memory (the B
// operand) for as long as the CTA stays in a limb.  One multiplication per
// input digit a and 16 inputs has N = 96: the six digits of 16 outputs, whose
// products land in the consecutive classes a .. a + 5 (16 columns each) of
// the accumulator, so a group of 16 outputs takes 6 K/16 instructions; a
// block's 32 signed sums take as many with N = 32.
#pragma once
#include <stdint.h>

#include "fiona_internal.h"

constexpr uint32_t kGemmDigits = 6, kGemmClasses = 2 * kGemmDigits - 1;
constexpr uint32_t kGemmRows = 128;         // coefficients per unit
constexpr uint32_t kGemmBlock = 32;         // outputs per block (two groups of 16)
constexpr uint32_t kGemmMaxInputs = 96;     // tensor memory: 6 * 48 columns of A + 192 of D
constexpr uint32_t kGemmMaxRaw = 64;        // raw terms per output
constexpr uint32_t kGemmEpilogueWarps = 16; // and one warp that issues the multiplications
constexpr uint32_t kGemmThreads = (kGemmEpilogueWarps + 1) * 32;
constexpr uint32_t kGemmNoGamma = 0xffffffffu;
constexpr uint32_t kGemmTestDigits = 1, kGemmTestFull = 2;  // the digits' barriers; the accumulators'

// one entry of G or W: output (in its chunk) and input; a raw entry's plaintext
struct GemmTerm {
    uint16_t out, in;
    uint32_t pt;      // raw: plaintext; signed: 1 for +1, 0 for -1
};

struct GemmArgs {
    const uint64_t *in, *pt;
    uint64_t *out;
    const LimbConst *limbs;
    int *err;
    const GemmTerm *raw, *sgn;   // by chunk
    const uint32_t *raw_off, *sgn_off;  // [n_chunks + 1]
    const uint32_t *gamma;       // per output: the scale group's plaintext, or kGemmNoGamma
    uint32_t N, L;               // L: limbs per poly in the buffers
    uint32_t limb0, n_limbs;
    uint32_t n_in, K, n_out;
    uint32_t chunk;              // outputs per chunk (a multiple of 32)
    uint32_t n_chunks;
    uint32_t units;              // chunks x limbs x coefficient tiles x polys
    uint64_t wait_ns;            // bound of every wait
    uint32_t test_flags;         // test only: barriers that expect an arrival too many (kGemmTest...)
    // 1, 2^8, 2^16, 2^24, read at run time: multiplications by literal powers
    // of two become several shifts and additions
    uint32_t c1, c8, c16, c24;
};

// dynamic shared memory of a CTA, byte offsets
struct GemmLayout {
    uint32_t group;   // one group's digits of G: 96 rows x K
    uint32_t w;       // one block's W: 32 rows x K
    uint32_t block;   // two groups, then W
    uint32_t bias, sbias, rowsum, wsum, gamma, sums, bars, total;
#if defined(__CUDACC__)
    __host__ __device__
#endif
    GemmLayout(uint32_t K, uint32_t chunk)
    {
        group = 16 * kGemmDigits * K * 2;
        w = kGemmBlock * K * 2;
        block = 2 * group + w;
        bias = block * (chunk / kGemmBlock);  // per output: raw bias (32 bytes), signed bias, row sums, gamma
        sbias = bias + chunk * 32;
        rowsum = sbias + chunk * 8;
        wsum = rowsum + chunk * 8;
        gamma = wsum + chunk * 4;
        sums = (gamma + chunk * 4 + 15) & ~15u;  // a block's signed sums: eight words per worker
        bars = sums + 8 * 8 * kGemmEpilogueWarps * 32;
        total = bars + 64;
    }
};

struct GemmSchedule {
    GemmArgs args{};          // device pointers (data pointers unset)
    size_t smem = 0;
    DeviceSchedule sched;
    uint32_t groups = 0;      // scale groups
    bool always = false;      // runs whatever its predicted time
};
