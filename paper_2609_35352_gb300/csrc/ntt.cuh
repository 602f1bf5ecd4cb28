// ntt.cuh -- the negacyclic transform machinery shared by the rescale
// (rescale.cu) and the plaintext encoder (encode.cu).
//
// Transform.  For a poly a of N = 2^n coefficients and psi a primitive 2N-th
// root of unity, the forward transform is A[k] = a(psi^(2 brv(k) + 1)),
// brv reversing the n bits of k: the radix-2 Cooley-Tukey stages (at the
// stage with m blocks, block i pairs elements at distance N / 2m with
// twiddle psi^brv(m + i)) from natural to bit-reversed order.  The inverse
// runs the Gentleman-Sande stages in the opposite order with psi^-brv(m + i)
// and then multiplies by N^-1.  The same passes serve residues mod q (psi a
// root mod q; the NTT of the RNS limbs) and, with cyclic decimation-in-time
// stages in the inverse's order (bit-reversed to natural), complex numbers (the
// canonical embedding of CKKS, whose slots are values of the plaintext at odd
// powers of exp(i pi / N)).
//
// Passes.  The stages are split between two passes over memory (N = R1 * R2,
// R1 = 2^floor(n/2)):
//   high pass  the first log2(R1) stages: for a fixed low index, the R1
//              elements hi * R2 + lo form one sub-transform; a CTA takes
//              tile / R1 of them (adjacent columns, so accesses coalesce);
//   low pass   the other stages, inside blocks of R2 consecutive elements;
//              a CTA takes tile / R2 blocks.
// A CTA's tile is 4096 elements in the high pass; in the low pass, whose CTAs
// also stage about one twiddle per element, it is the same rows of eight polys
// (4096 elements, 512 twiddles) for the transforms mod q, or of one poly where
// there are few, and 2048 elements of one for the complex ones.  A thread
// handles 16 elements (8 of a tile of 512).
// A pass runs its stages in rounds of up to 4: in a round each thread holds
// the 2^K elements of one group in registers, spaced by the round's smallest
// distance, and applies the round's K stages to them (a group needs 2^K - 1
// twiddles).  Rounds hand over through shared memory ([sub-transform]
// [position], one element of padding per row against bank conflicts); the
// first and last rounds of a pass read and write global memory directly
// wherever their access pattern coalesces.  The CTA's twiddles are copied to
// shared memory (cp.async) while its data loads are in flight.  Everything is
// instantiated per log2 N, so all index arithmetic is constant-folded.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fiona_ntt {

constexpr int kLogTileMax = 12;  // at most 4096 elements per CTA
constexpr int kLogNMin = 10, kLogNMax = 17;  // the ring dimensions a context accepts

// B bytes (16, or 8) global -> shared, asynchronous
template <int B>
__device__ __forceinline__ void cp_async(void *smem, const void *gmem)
{
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
    if constexpr (B == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}

// ---------------------------------------------------------------------------
// Residues mod q < 2^60 in 64-bit words.
// ---------------------------------------------------------------------------
// x - c if that is not negative, else x (x - c within a signed word: every
// use has x, c < 12q and |x - c| < 7q < 2^63; the sign is one test of the
// high half)
__device__ __forceinline__ uint64_t csub(uint64_t x, uint64_t c)
{
    const int64_t d = (int64_t)(x - c);
    return d < 0 ? x : (uint64_t)d;
}

// x in [0, 6q) -> canonical
__device__ __forceinline__ uint64_t canon6(uint64_t x, uint64_t q) { return csub(csub(csub(x, 4 * q), 2 * q), q); }

// x mod q for any 64-bit x: floor(x * mu64 / 2^64), mu64 = floor(2^64 / q),
// is floor(x / q) or one less
__device__ __forceinline__ uint64_t reduce_any(uint64_t x, uint64_t q, uint64_t mu64)
{
    return csub(x - __umul64hi(x, mu64) * q, q);
}

// A constant w of a limb (a twiddle, N^-1, q_j^-1): w and v = w 2^32 mod q,
// and their quotients by 2q, om = floor(2^32 w / 2q) and ov = floor(2^32 v /
// 2q), both below 2^31.
struct __align__(16) Twiddle {
    ulonglong2 wv;  // (w, v)
    uint2 om;       // (om, ov)
};
struct TwiddleTable {  // a limb's table in global memory
    const ulonglong2 *wv;
    const uint2 *om;
};
struct TwiddleStage {  // a pass's twiddles in shared memory
    ulonglong2 *wv;
    uint2 *om;
    __device__ __forceinline__ Twiddle operator[](uint32_t i) const { return Twiddle{wv[i], om[i]}; }
};

// x * w mod q for any 64-bit x = xh 2^32 + xl, lazily: V = xl w + xh v is
// congruent to x w; with k = floor((xl om + xh ov) / 2^32),
//   V / 2q - 3 < k <= V / 2q
// (om and ov fall short of their exact values by less than 1 each, so the
// sum by less than xl + xh < 2^33; the floor takes less than 1 more), and
// r = V - k 2q, computed modulo 2^64, lies in [0, 6q), below 2^63.  The sum
// does not wrap (each product is below 2^63), and k fits in 32 bits: that is
// what the quotient by 2q is for.
// Five 32x32 -> 64-bit products and three 32-bit ones.  Shoup's product with
// one precomputed quotient floor(2^64 w / q) takes five (two of them for the
// high half only) and four.  The FMA-heavy pipe bounds every transform here,
// and on sm_103a a 64-bit product holds it for 4 cycles a warp, a 32-bit one
// for 2.  Measured in a register-only chain of radix-16 groups (GB300, 16
// warps an SM): 36.0 cycles a butterfly and warp scheduler against 42.4, the
// pipe 85-89% busy in both.  The product by k is added last and by itself:
// with the three wide products in one chain of multiply-adds it measured
// 39.7; written without the explicit word operations, 37-40.
__device__ __forceinline__ uint64_t mul_twiddle(uint64_t x, const Twiddle &t, uint64_t q)
{
    const uint32_t xl = (uint32_t)x, xh = (uint32_t)(x >> 32);
    const uint64_t n = 0 - 2 * q;
    uint64_t m, p, k2, r;
    uint32_t hi;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(m) : "r"(xl), "r"(t.om.x));
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(m) : "r"(xh), "r"(t.om.y));
    const uint32_t k = (uint32_t)(m >> 32);
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(xl), "r"((uint32_t)t.wv.x));
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(p) : "r"(xh), "r"((uint32_t)t.wv.y));
    hi = (uint32_t)(p >> 32);
    asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(hi) : "r"(xl), "r"((uint32_t)(t.wv.x >> 32)));
    asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(hi) : "r"(xh), "r"((uint32_t)(t.wv.y >> 32)));
    asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(hi) : "r"(k), "r"((uint32_t)(n >> 32)));
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(k2) : "r"(k), "r"((uint32_t)n));
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"((uint32_t)p), "r"(hi));
    return r + k2;
}

// Modular butterflies.  Values between stages:
//   forward, general   in [0, 12q): x is brought below 6q before each
//                      butterfly (x + t, x - t + 6q with t in [0, 6q));
//   forward, FAST      (q < 2^56, inputs below 8q) no reduction at all: each
//                      stage adds less than 6q to the bound, so after at most
//                      17 stages values stay below 110q < 2^63;
//   inverse            in [0, 6q): x + y is brought below 6q, and
//                      x - y + 6q is only multiplied.
// A pass stages its twiddles in shared memory as two arrays (16 and 8 bytes
// an entry).
template <bool FAST>
struct ModArith {
    typedef uint64_t T;
    typedef Twiddle W;
    static constexpr size_t w_bytes = 24;
    static constexpr bool kCyclic = false;
    typedef TwiddleTable Table;
    typedef TwiddleStage Staged;
    __device__ __forceinline__ static Staged staged(uint8_t *raw, int entries)
    {
        return Staged{reinterpret_cast<ulonglong2 *>(raw), reinterpret_cast<uint2 *>(raw + 16 * (size_t)entries)};
    }
    __device__ __forceinline__ static void stage(const Staged &s, uint32_t i, const Table &t, uint32_t k)
    {
        cp_async<16>(&s.wv[i], &t.wv[k]);
        cp_async<8>(&s.om[i], &t.om[k]);
    }
    uint64_t q;
    __device__ __forceinline__ void ct(T &x, T &y, const W &w) const
    {
        const uint64_t a = FAST ? x : csub(x, 6 * q);
        const uint64_t t = mul_twiddle(y, w, q);
        x = a + t;
        y = a + 6 * q - t;
    }
    __device__ __forceinline__ void gs(T &x, T &y, const W &w) const
    {
        const uint64_t a = x, b = y;
        x = csub(a + b, 6 * q);
        y = mul_twiddle(a + 6 * q - b, w, q);
    }
};

// Complex numbers in fp64 (re, im); twiddles are (cos, sin) pairs.  These
// transforms are cyclic (kCyclic): the pair at distance h takes the twiddle
// exp(-i pi (pos mod h) / h), the same for every block, which sits at entry
// h + (pos mod h) of a table shared by both passes.  A butterfly x + w y, x - w y
// is six fused operations: x + w y by four, and 2x less that by two.
struct CplxArith {
    typedef double2 T;
    typedef double2 W;
    static constexpr size_t w_bytes = 16;
    static constexpr bool kCyclic = true;
    typedef const double2 *Table;
    typedef double2 *Staged;
    __device__ __forceinline__ static Staged staged(uint8_t *raw, int) { return reinterpret_cast<double2 *>(raw); }
    __device__ __forceinline__ static void stage(Staged s, uint32_t i, Table t, uint32_t k) { cp_async<16>(&s[i], &t[k]); }
    __device__ __forceinline__ static double2 mul(double2 a, double2 b)
    {
        return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
    }
    __device__ __forceinline__ static void butterfly(T &x, T &y, W w)
    {
        const double re = fma(-y.y, w.y, fma(y.x, w.x, x.x)), im = fma(y.x, w.y, fma(y.y, w.x, x.y));
        y = make_double2(fma(2.0, x.x, -re), fma(2.0, x.y, -im));
        x = make_double2(re, im);
    }
    // x - w y on its own, eight operations: one rounding less.  Taken in the last
    // stage of each pass, and from 2^15 slots on in the last two of the high
    // pass: the transform's error is then below that of eight-operation stages
    // throughout at every ring size (relative 2-norm against extended precision,
    // complex slots: 2.11e-16 against 2.20e-16 at 2^9, 2.70 against 2.71 at 2^14,
    // 2.79 against 2.81 at 2^15, 2.875 against 2.887 at 2^16; with one stage only
    // 2.896 there).  Embedding 93 vectors of 2^15: 0.326 ms, 0.322 with one
    // stage, 0.315 with none.
    __device__ __forceinline__ static void butterfly_direct(T &x, T &y, W w)
    {
        const double2 a = x, b = y;
        x = make_double2(fma(-b.y, w.y, fma(b.x, w.x, a.x)), fma(b.x, w.y, fma(b.y, w.x, a.y)));
        y = make_double2(fma(b.y, w.y, fma(-b.x, w.x, a.x)), fma(-b.x, w.y, fma(-b.y, w.x, a.y)));
    }
    // w = 1 and w = -i
    __device__ __forceinline__ static void butterfly_1(T &x, T &y)
    {
        const double2 a = x, b = y;
        x = make_double2(a.x + b.x, a.y + b.y);
        y = make_double2(a.x - b.x, a.y - b.y);
    }
    __device__ __forceinline__ static void butterfly_i(T &x, T &y)
    {
        const double2 a = x, b = y;
        x = make_double2(a.x + b.y, a.y - b.x);
        y = make_double2(a.x - b.y, a.y + b.x);
    }
};

// ---------------------------------------------------------------------------
// Compile-time geometry
// ---------------------------------------------------------------------------
template <int LOGN>
struct Shape {
    static constexpr int n1 = LOGN / 2;
    static constexpr int lt = LOGN < kLogTileMax ? LOGN : kLogTileMax;  // log2(tile)
    static constexpr int ltiles = LOGN - lt;                            // log2(tiles per transform)
};

// A pass over a tile: 2^LSUBS sub-transforms of 2^S positions, in rounds,
// 2^LTILES tiles per transform, 16 elements per thread (at least 64 threads).
// With LPOLYS > 0 (low pass) the sub-transforms are the same 2^lrows rows of
// 2^LPOLYS polys: sub = poly << lrows | row, and the polys share their
// twiddles.
template <int S, int LSUBS, bool HIGH, int LTILES, int LPOLYS = 0>
struct PassShape {
    static constexpr int s = S, lsubs = LSUBS, subs = 1 << LSUBS;
    static constexpr int lpolys = LPOLYS, polys = 1 << LPOLYS, lrows = LSUBS - LPOLYS, rows = 1 << lrows;
    static constexpr int tile = 1 << (S + LSUBS);
    static constexpr int ltiles = LTILES;
    static constexpr uint32_t threads = tile / 16 < 64 ? 64 : tile / 16;
    static constexpr int pitch = (1 << S) + 1;
    static constexpr int nr = (S + 3) / 4;
    __host__ __device__ static constexpr int K(int r) { return S / nr + (r < S % nr ? 1 : 0); }
    __host__ __device__ static constexpr int J0(int r) { return r == 0 ? 0 : J0(r - 1) + K(r - 1); }
    static constexpr bool high = HIGH;
    // shared memory: the staged twiddles (2^s entries for the high pass, at
    // most one per element of a poly's rows for the low pass), then the
    // padded tile
    template <class A>
    __host__ __device__ static constexpr int entries()
    {
        return HIGH || A::kCyclic ? 1 << S : 1 << (S + lrows);
    }
    template <class A>
    __host__ __device__ static constexpr size_t smem_bytes()
    {
        return A::w_bytes * entries<A>() + sizeof(typename A::T) * subs * pitch;
    }
};

template <int LOGN>
using HighPass = PassShape<Shape<LOGN>::n1, Shape<LOGN>::lt - Shape<LOGN>::n1, true, Shape<LOGN>::ltiles>;
// the low pass: a tile of half the high pass's, but at least one block
template <int LOGN>
struct LowShape {
    static constexpr int s = LOGN - Shape<LOGN>::n1;
    static constexpr int lt = Shape<LOGN>::lt - 1 > s ? Shape<LOGN>::lt - 1 : s;
};
template <int LOGN>
using LowPass = PassShape<LowShape<LOGN>::s, LowShape<LOGN>::lt - LowShape<LOGN>::s, false, LOGN - LowShape<LOGN>::lt>;

// The low pass of several polys at once (the transforms mod q): a tile of
// 4096 elements, kPolys polys of 4096 / kPolys.  A low-pass CTA needs one
// twiddle (24 bytes) per element of its rows, read through L2 and staged by
// its threads; sharing them between the polys of a batch divides both that
// traffic and its instructions by kPolys, and leaves room for 32 warps an SM
// (45 KB a CTA of 256 threads).  Measured on GB300, 192 polys of 2^16, 12
// limbs: the rescale 1.488 ms with 4 polys a CTA, 1.410 with 8.
constexpr int kLogPolys = 3, kPolys = 1 << kLogPolys;
// LP = kLogPolys, or fewer polys with the same rows (and the same table)
template <int LOGN, int LP = kLogPolys>
using LowPassPolys = PassShape<LOGN - Shape<LOGN>::n1, kLogTileMax - (LOGN - Shape<LOGN>::n1) - kLogPolys + LP, false,
                               LOGN - kLogTileMax + kLogPolys, LP>;

// Group g of round R: sub-transform `sub`, and the element positions
// (hi << (lD + K)) + (i << lD) + lo, i < 2^K.  High pass: sub-transforms
// fastest (adjacent columns); low pass: lo fastest (adjacent elements).
template <class PS, int R>
struct Group {
    static constexpr int K = PS::K(R), J0 = PS::J0(R), LD = PS::s - J0 - K;
    static constexpr int groups = PS::tile >> K;
    static constexpr int per_thread = (groups + (int)PS::threads - 1) / (int)PS::threads;
    uint32_t sub, hi, lo;
    __device__ __forceinline__ explicit Group(uint32_t g)
    {
        if (PS::high) {
            sub = g & (PS::subs - 1);
            const uint32_t rest = g >> PS::lsubs;
            lo = rest & ((1u << LD) - 1);
            hi = rest >> LD;
        } else {
            lo = g & ((1u << LD) - 1);
            const uint32_t rest = g >> LD;
            sub = rest & (PS::subs - 1);
            hi = rest >> PS::lsubs;
        }
    }
    __device__ __forceinline__ uint32_t pos(int i) const { return (hi << (LD + K)) + ((uint32_t)i << LD) + lo; }
    // twiddle of local stage J0 + k, block b of the group, in the staged layout
    __device__ __forceinline__ uint32_t tw(int k, int b) const
    {
        const int j = J0 + k;
        if (PS::high) return (1u << j) + (hi << k) + b;
        return ((PS::rows << j) - PS::rows) + (((hi << k) + b) << PS::lrows) + (sub & (PS::rows - 1));
    }
};

template <class PS, int R, int k, bool INV, class A>
__device__ __forceinline__ void group_stage(typename A::T (&x)[1 << PS::K(R)], const Group<PS, R> &G,
                                            const typename A::Staged &stw, const A &ar)
{
    constexpr int K = PS::K(R), h = 1 << (K - 1 - k);
#pragma unroll
    for (int b = 0; b < (1 << k); ++b) {
        const typename A::W w = stw[G.tw(k, b)];
#pragma unroll
        for (int a = 0; a < h; ++a) {
            if (INV)
                ar.gs(x[b * 2 * h + a], x[b * 2 * h + a + h], w);
            else
                ar.ct(x[b * 2 * h + a], x[b * 2 * h + a + h], w);
        }
    }
}

// the cyclic stages of a group, smallest distance first (the order of the
// inverse); in the first round (LD = 0) the twiddles 1 and -i take plain
// additions
template <class PS, int R, class A>
__device__ __forceinline__ void cyclic_stages(typename A::T (&x)[1 << PS::K(R)], const Group<PS, R> &G,
                                              const typename A::Staged &stw)
{
    constexpr int K = PS::K(R), LD = Group<PS, R>::LD;
    // the last stages of the pass by direct butterflies (CplxArith)
    constexpr int direct = PS::high && PS::s + PS::lsubs + PS::ltiles >= 15 ? 2 : 1;
#pragma unroll
    for (int t = 0; t < K; ++t)
#pragma unroll
        for (int m = 0; m < (1 << t); ++m) {
            constexpr bool first = LD == 0;
            const bool one = first && m == 0, minus_i = first && t > 0 && m == (1 << t) / 2;
            typename A::W w;
            if (!one && !minus_i) w = stw[(1u << (LD + t)) + ((uint32_t)m << LD) + G.lo];
#pragma unroll
            for (int b = m; b < (1 << K); b += 2 << t) {
                if (one)
                    A::butterfly_1(x[b], x[b + (1 << t)]);
                else if (minus_i)
                    A::butterfly_i(x[b], x[b + (1 << t)]);
                else if (R == 0 && t >= K - direct)
                    A::butterfly_direct(x[b], x[b + (1 << t)], w);
                else
                    A::butterfly(x[b], x[b + (1 << t)], w);
            }
        }
}

template <class PS, int R, bool INV, class A>
__device__ __forceinline__ void group_stages(typename A::T (&x)[1 << PS::K(R)], const Group<PS, R> &G,
                                             const typename A::Staged &stw, const A &ar)
{
    constexpr int K = PS::K(R);
    if constexpr (A::kCyclic) {
        static_assert(INV, "cyclic transforms: smallest distance first");
        cyclic_stages<PS, R, A>(x, G, stw);
    } else if constexpr (!INV) {
        group_stage<PS, R, 0, false>(x, G, stw, ar);
        if constexpr (K > 1) group_stage<PS, R, 1, false>(x, G, stw, ar);
        if constexpr (K > 2) group_stage<PS, R, 2, false>(x, G, stw, ar);
        if constexpr (K > 3) group_stage<PS, R, 3, false>(x, G, stw, ar);
    } else {
        if constexpr (K > 3) group_stage<PS, R, 3, true>(x, G, stw, ar);
        if constexpr (K > 2) group_stage<PS, R, 2, true>(x, G, stw, ar);
        if constexpr (K > 1) group_stage<PS, R, 1, true>(x, G, stw, ar);
        group_stage<PS, R, 0, true>(x, G, stw, ar);
    }
}

// Whether sub-transform `sub` is one of the `np` polys a CTA has (the last
// group of a batch may have fewer than PS::polys: their rows take part in
// nothing).
template <class PS>
__device__ __forceinline__ bool present(uint32_t sub, uint32_t np)
{
    return PS::lpolys == 0 || (sub >> PS::lrows) < np;
}

// One round: every group of this thread is loaded (ld(sub, pos)), then
// `between()` runs (once, on every thread), then the groups are transformed
// and stored (st(sub, pos, value)).
template <class PS, int R, bool INV, class A, class Ld, class Between, class St>
__device__ __forceinline__ void round(const typename A::Staged &stw, const A &ar, uint32_t np, Ld ld, Between between,
                                      St st)
{
    using Gr = Group<PS, R>;
    constexpr int P = Gr::per_thread, E = 1 << Gr::K;
    typename A::T x[P][E];
#pragma unroll
    for (int gi = 0; gi < P; ++gi) {
        const uint32_t g = threadIdx.x + gi * PS::threads;
        if (Gr::groups % PS::threads == 0 || g < Gr::groups) {
            const Gr G(g);
            if (present<PS>(G.sub, np))
#pragma unroll
                for (int i = 0; i < E; ++i) x[gi][i] = ld(G.sub, G.pos(i));
        }
    }
    between();
#pragma unroll
    for (int gi = 0; gi < P; ++gi) {
        const uint32_t g = threadIdx.x + gi * PS::threads;
        if (Gr::groups % PS::threads == 0 || g < Gr::groups) {
            const Gr G(g);
            if (present<PS>(G.sub, np)) {
                group_stages<PS, R, INV>(x[gi], G, stw, ar);
#pragma unroll
                for (int i = 0; i < E; ++i) st(G.sub, G.pos(i), x[gi][i]);
            }
        }
    }
}

// the rounds from R up to (excluding) REND, through shared memory
template <class PS, int R, int REND, bool INV, class A>
__device__ __forceinline__ void middle_rounds(typename A::T *sm, const typename A::Staged &stw, const A &ar, uint32_t np)
{
    if constexpr (R != REND) {
        round<PS, R, INV>(
            stw, ar, np, [&](uint32_t sub, uint32_t pos) { return sm[sub * PS::pitch + pos]; }, [] {},
            [&](uint32_t sub, uint32_t pos, typename A::T v) { sm[sub * PS::pitch + pos] = v; });
        __syncthreads();
        middle_rounds<PS, (INV ? R - 1 : R + 1), REND, INV>(sm, stw, ar, np);
    }
}

// The tables.  Entry k >= 1 of a transform's twiddles is psi^brv(k) (forward)
// or psi^-brv(k) (inverse); the stage with m blocks uses entries m .. 2m - 1.
// The high pass needs entries [0, R1): the entry of its local stage j for
// position pos is 2^j + (pos >> (s - j)), for every sub-transform.  Row `row`
// of the low pass needs ((R1 + row) << j) + t for its local stages j < s and
// t < 2^j, each entry of [R1, N) used by one row; they are stored in the
// order in which a CTA stages them, so that staging is a plain copy: the
// rows of a CTA's tile together, stage j's entries from (rows << j) - rows
// on, t-major ([t][row]: adjacent rows read adjacent words of shared memory).
// (With the entries at their index k and the order made while staging, that
// took 27% of the forward low pass's instructions.)  low_place is the place of
// entry k for tiles of 2^lrows rows.
inline uint32_t low_place(uint32_t k, uint32_t n1, uint32_t s, uint32_t lrows)
{
    if (k >> n1 == 0) return k;
    uint32_t j = 0;
    while (k >> (n1 + j + 1)) ++j;
    const uint32_t row = (k >> j) - (1u << n1), t = k & ((1u << j) - 1);
    const uint32_t tile = row >> lrows, r = row & ((1u << lrows) - 1);
    return (1u << n1) + ((tile * ((1u << s) - 1)) << lrows) + (((1u << j) - 1) << lrows) + (t << lrows) + r;
}

// Stage the pass's twiddles (cp.async; waited by wait_twiddles); `first` is
// the low pass's first row
template <int LOGN, class PS, class A>
__device__ __forceinline__ void stage_twiddles(const typename A::Staged &stw, const typename A::Table &tab, uint32_t first)
{
    constexpr bool whole = PS::high || A::kCyclic;  // entries [0, 2^s)
    constexpr uint32_t cnt = whole ? 1u << PS::s : (uint32_t)PS::rows * ((1u << PS::s) - 1);
    const uint32_t base = whole ? 0 : (1u << Shape<LOGN>::n1) + first * ((1u << PS::s) - 1);
#pragma unroll
    for (uint32_t e = 0; e < cnt; e += PS::threads)
        if (e + PS::threads <= cnt || e + threadIdx.x < cnt) A::stage(stw, e + threadIdx.x, tab, base + e + threadIdx.x);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}

__device__ __forceinline__ void wait_twiddles()
{
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
}

// the same for the element e0 + t of a sweep below (a poly's rows are a
// multiple of the threads)
template <class PS>
__device__ __forceinline__ bool has(uint32_t e0, uint32_t np)
{
    static_assert(PS::lpolys == 0 || (1 << (PS::s + PS::lrows)) % PS::threads == 0, "whole steps per poly");
    return PS::lpolys == 0 || (e0 >> (PS::s + PS::lrows)) < np;
}

// A coalesced sweep over the tile's elements e = e0 + t (tile / threads per
// thread; e0 a constant multiple of the thread count, t the thread): every
// load first, then every store.
template <class PS, class T, class Ld, class St>
__device__ __forceinline__ void sweep(uint32_t np, Ld ld, St st)
{
    constexpr int P = (PS::tile + (int)PS::threads - 1) / (int)PS::threads;
    T v[P];
#pragma unroll
    for (int i = 0; i < P; ++i)
        if ((PS::tile % PS::threads == 0 || threadIdx.x + i * PS::threads < PS::tile) && has<PS>(i * PS::threads, np))
            v[i] = ld(i * PS::threads, threadIdx.x);
#pragma unroll
    for (int i = 0; i < P; ++i)
        if ((PS::tile % PS::threads == 0 || threadIdx.x + i * PS::threads < PS::tile) && has<PS>(i * PS::threads, np))
            st(i * PS::threads, threadIdx.x, v[i]);
}

// the padded position of element e0 + t of a tile in shared memory
template <class PS>
__device__ __forceinline__ uint32_t padded(uint32_t e0, uint32_t t)
{
    if constexpr (PS::threads % (1u << PS::s) == 0)  // whole rows per step
        return ((e0 >> PS::s) + (t >> PS::s)) * PS::pitch + (t & ((1u << PS::s) - 1));
    else
        return ((e0 + t) >> PS::s) * PS::pitch + ((e0 + t) & ((1u << PS::s) - 1));
}

// shared memory of a pass: staged twiddles, then the tile
template <class PS, class A>
struct Smem {
    typename A::Staged stw;
    typename A::T *sm;
    __device__ __forceinline__ explicit Smem(uint8_t *raw)
        : stw(A::staged(raw, PS::template entries<A>())),
          sm(reinterpret_cast<typename A::T *>(raw + A::w_bytes * PS::template entries<A>()))
    {
    }
};

// ---------------------------------------------------------------------------
// Pass drivers.  `first` is the tile's first column (high) or row (low);
// the callbacks address the tile by (sub, pos), or by the element index e =
// sub * 2^s + pos of a coalesced sweep.  Low passes take the pass shape and
// the polys the CTA has.
// ---------------------------------------------------------------------------

// forward high pass: the first round loads directly (gload), the last stores
// directly (gstore)
template <int LOGN, class A, class GLoad, class GStore>
__device__ __forceinline__ void fwd_high_pass(uint8_t *raw, const typename A::Table &tab, uint32_t first, const A &ar,
                                              GLoad gload, GStore gstore)
{
    using PS = HighPass<LOGN>;
    Smem<PS, A> S(raw);
    typename A::T *sm = S.sm;
    stage_twiddles<LOGN, PS, A>(S.stw, tab, first);
    auto sload = [&](uint32_t sub, uint32_t pos) { return sm[sub * PS::pitch + pos]; };
    auto sstore = [&](uint32_t sub, uint32_t pos, typename A::T v) { sm[sub * PS::pitch + pos] = v; };
    if constexpr (PS::nr == 1) {
        round<PS, 0, false>(S.stw, ar, 1, gload, wait_twiddles, gstore);
    } else {
        round<PS, 0, false>(S.stw, ar, 1, gload, wait_twiddles, sstore);
        __syncthreads();
        middle_rounds<PS, 1, PS::nr - 1, false>(sm, S.stw, ar, 1);
        round<PS, PS::nr - 1, false>(S.stw, ar, 1, sload, [] {}, gstore);
    }
}

// forward low pass: the first round (lo fastest) loads directly; the last
// round goes through shared memory to a coalesced sweep epi(value of e0, t), every
// value read by then (`pre()` runs before the first round)
template <int LOGN, class PS, class A, class Pre, class GLoad, class Epi>
__device__ __forceinline__ void fwd_low_pass(uint8_t *raw, const typename A::Table &tab, uint32_t first, const A &ar,
                                             uint32_t np, Pre pre, GLoad gload, Epi epi)
{
    Smem<PS, A> S(raw);
    typename A::T *sm = S.sm;
    stage_twiddles<LOGN, PS, A>(S.stw, tab, first);
    pre();
    auto sstore = [&](uint32_t sub, uint32_t pos, typename A::T v) { sm[sub * PS::pitch + pos] = v; };
    round<PS, 0, false>(S.stw, ar, np, gload, wait_twiddles, sstore);
    __syncthreads();
    middle_rounds<PS, 1, PS::nr, false>(sm, S.stw, ar, np);
    epi([&](uint32_t e0, uint32_t t) { return sm[padded<PS>(e0, t)]; });
}

// inverse low pass: a coalesced sweep in (sweep_load(e0, t)), the rounds, the
// last round (lo fastest) stores directly
template <int LOGN, class PS, class A, class SLoad, class GStore>
__device__ __forceinline__ void inv_low_pass(uint8_t *raw, const typename A::Table &tab, uint32_t first, const A &ar,
                                             uint32_t np, SLoad sweep_load, GStore gstore)
{
    Smem<PS, A> S(raw);
    typename A::T *sm = S.sm;
    stage_twiddles<LOGN, PS, A>(S.stw, tab, first);
    sweep<PS, typename A::T>(np, sweep_load, [&](uint32_t e0, uint32_t t, typename A::T v) { sm[padded<PS>(e0, t)] = v; });
    wait_twiddles();
    middle_rounds<PS, PS::nr - 1, 0, true>(sm, S.stw, ar, np);
    round<PS, 0, true>(
        S.stw, ar, np, [&](uint32_t sub, uint32_t pos) { return sm[sub * PS::pitch + pos]; }, [] {}, gstore);
}

// inverse high pass: the first round (sub-transforms fastest) loads
// directly, the last stores directly
template <int LOGN, class A, class GLoad, class GStore>
__device__ __forceinline__ void inv_high_pass(uint8_t *raw, const typename A::Table &tab, uint32_t first, const A &ar,
                                              GLoad gload, GStore gstore)
{
    using PS = HighPass<LOGN>;
    Smem<PS, A> S(raw);
    typename A::T *sm = S.sm;
    stage_twiddles<LOGN, PS, A>(S.stw, tab, first);
    auto sload = [&](uint32_t sub, uint32_t pos) { return sm[sub * PS::pitch + pos]; };
    auto sstore = [&](uint32_t sub, uint32_t pos, typename A::T v) { sm[sub * PS::pitch + pos] = v; };
    if constexpr (PS::nr == 1) {
        round<PS, 0, true>(S.stw, ar, 1, gload, wait_twiddles, gstore);
    } else {
        round<PS, PS::nr - 1, true>(S.stw, ar, 1, gload, wait_twiddles, sstore);
        __syncthreads();
        middle_rounds<PS, PS::nr - 2, 0, true>(sm, S.stw, ar, 1);
        round<PS, 0, true>(S.stw, ar, 1, sload, [] {}, gstore);
    }
}

// Per-limb modular tables, in device memory (built on the host once per
// context; the tables follow the array of these).
struct NttLimb {
    TwiddleTable fwd;        // [N]: psi^brv(k)
    TwiddleTable inv;        // [N]: psi^-brv(k)
    const Twiddle *qinv;     // [L]: q_j^-1 mod q for j > this limb, else 0
    uint64_t q;
    uint64_t mu64;           // floor(2^64 / q)
    Twiddle ninv;            // N^-1 mod q
};

// host: log2 of a power of two
inline uint32_t log2u(uint32_t N)
{
    uint32_t n = 0;
    while ((1u << n) < N) ++n;
    return n;
}

// host: bit reversal of the low `bits` bits
inline uint32_t bit_reverse(uint32_t k, uint32_t bits)
{
    uint32_t r = 0;
    for (uint32_t b = 0; b < bits; ++b) r = (r << 1) | ((k >> b) & 1u);
    return r;
}

}  // namespace fiona_ntt
