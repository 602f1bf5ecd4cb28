// rescale.cu -- the rescale that follows the layer: every output poly is
// divided by the last prime of its level (Sec. 2.2 "Homomorphic Operations":
// a PMult raises the scale and a rescale restores it; Sec. 4.2 "Combining
// the Signed and Raw Routes": one rescale per output).  For a poly y with
// limbs y_0..y_{Lc-1} in NTT form:
//   r    = coefficients of y_{Lc-1}       (inverse NTT mod q_{Lc-1})
//   y'_l = (y_l - NTT_l(r mod q_l)) * q_{Lc-1}^{-1}  mod q_l,   l < Lc-1,
// the quotient of the CRT value Y by q_{Lc-1} rounded down; rounded to the
// nearest (the variant that adds h = floor(q_{Lc-1} / 2) to Y), r becomes
// r' = (r + h) mod q_{Lc-1} and the subtracted poly r' - h (mod q_l).
// NTT form: A[k] = a(psi^(2 brv(k) + 1)) mod q, psi the least primitive
// 2N-th root of unity mod q (the transform and its passes: ntt.cuh).
//
// The rescale is four launches on the caller's stream: the two inverse passes
// on the last limb of every poly (in place: it becomes the coefficients r,
// canonical), then the two forward passes of every other limb; the first
// reads r and reduces it mod q_l (unless r < 4 q_l already, with every
// q_l < 2^56: then the reduction-free butterflies take it as it is), the
// second applies the subtraction and the product by q_{Lc-1}^{-1}.  The whole
// last limb must be known before any limb can be finished, so the rescale
// cannot share a launch with the layer's kernels, whose CTAs each see one
// tile of coefficients.
//
// What bounds it: the FMA-heavy pipe (64-bit products, 4 cycles a warp), which
// ncu shows 76% busy in the forward high pass and 69% in the low one, whose
// epilogue also reads y.  Measured on GB300 (192 polys of 2^16, 12 -> 11
// limbs): 1.728 ms with Shoup's product and one poly a low-pass CTA, 1.410 ms with
// the two-word twiddles of ntt.cuh, their tables in staging order and eight polys;
// its HBM bytes take 0.34 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "fiona_internal.h"
#include "ntt.cuh"

using namespace fiona_ntt;

namespace {

typedef unsigned __int128 u128;

struct Args {
    uint64_t *polys;   // [count][Lc][N]
    uint64_t *out;     // [count][Lc-1][N]
    const NttLimb *T;
    uint32_t count;
    uint32_t Lc;
    uint32_t round;    // 1: nearest quotient (add h = floor(q_{Lc-1} / 2))
};

// ---------------------------------------------------------------------------
// The four launches.  blockIdx.x = transform * tiles + tile; the transforms
// are the polys (inverse high pass), poly * (Lc - 1) + limb (forward high
// pass), and for the low passes, whose CTAs take the same rows of kPolys
// polys or of one (many_polys), group of polys (inverse) or group * (Lc - 1) +
// limb (forward).
// ---------------------------------------------------------------------------

// inverse, low stages, on the last limb in place
template <int LOGN, int LP>
__global__ void __launch_bounds__(LowPassPolys<LOGN, LP>::threads, LP ? 3 : 12) k_inv_low(Args A)
{
    using PS = LowPassPolys<LOGN, LP>;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t tile = blockIdx.x & ((1u << PS::ltiles) - 1), p0 = (blockIdx.x >> PS::ltiles) << PS::lpolys;
    const uint32_t first = tile << PS::lrows;
    const size_t stride = (size_t)A.Lc << LOGN;
    uint64_t *g = A.polys + p0 * stride + ((size_t)(A.Lc - 1) << LOGN) + ((size_t)first << PS::s);
    const NttLimb &Tl = A.T[A.Lc - 1];
    constexpr int le = PS::s + PS::lrows;  // log2 elements per poly
    inv_low_pass<LOGN, PS>(
        smem_raw, Tl.inv, first, ModArith<false>{Tl.q}, A.count - p0,
        [&](uint32_t e0, uint32_t t) { return g[(e0 >> le) * stride + (e0 & ((1u << le) - 1)) + t]; },
        [&](uint32_t sub, uint32_t pos, uint64_t v) {
            g[(sub >> PS::lrows) * stride + ((sub & (PS::rows - 1)) << PS::s) + pos] = v;
        });
}

// inverse, high stages: stores r = N^-1 x, canonical
template <int LOGN>
__global__ void __launch_bounds__(HighPass<LOGN>::threads, 3) k_inv_high(Args A)
{
    using PS = HighPass<LOGN>;
    constexpr uint32_t R2 = 1u << (LOGN - Shape<LOGN>::n1);
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t tile = blockIdx.x & ((1u << PS::ltiles) - 1), p = blockIdx.x >> PS::ltiles;
    const uint32_t first = tile << PS::lsubs;
    uint64_t *g = A.polys + ((size_t)p * A.Lc + (A.Lc - 1)) * (1u << LOGN) + first;
    const NttLimb &Tl = A.T[A.Lc - 1];
    const uint64_t q = Tl.q;
    const Twiddle ninv = Tl.ninv;
    const uint64_t h = A.round ? q / 2 : 0;
    inv_high_pass<LOGN>(smem_raw, Tl.inv, first, ModArith<false>{q},
                        [&](uint32_t sub, uint32_t pos) { return g[(size_t)pos * R2 + sub]; },
                        [&](uint32_t sub, uint32_t pos, uint64_t v) {
                            g[(size_t)pos * R2 + sub] = csub(canon6(mul_twiddle(v, ninv, q), q) + h, q);
                        });
}

// forward, high stages: r (the last limb's coefficients), reduced mod q_l
// unless FAST, into out
template <int LOGN, bool FAST>
__global__ void __launch_bounds__(HighPass<LOGN>::threads, 3) k_fwd_high(Args A)
{
    using PS = HighPass<LOGN>;
    constexpr uint32_t R2 = 1u << (LOGN - Shape<LOGN>::n1);
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t tile = blockIdx.x & ((1u << PS::ltiles) - 1), tr = blockIdx.x >> PS::ltiles;
    const uint32_t p = tr / (A.Lc - 1), l = tr % (A.Lc - 1);
    const uint32_t first = tile << PS::lsubs;
    const uint64_t *g = A.polys + ((size_t)p * A.Lc + (A.Lc - 1)) * (1u << LOGN) + first;
    uint64_t *o = A.out + (size_t)tr * (1u << LOGN) + first;
    const NttLimb &Tl = A.T[l];
    const uint64_t q = Tl.q, mu = Tl.mu64;
    // rounding: subtract h mod q_l, as + (q_l - h mod q_l); the loaded value
    // then stays below 5 q_l (FAST) or 2 q_l
    const uint64_t hq = A.round ? q - reduce_any(A.T[A.Lc - 1].q / 2, q, mu) : 0;
    fwd_high_pass<LOGN>(
        smem_raw, Tl.fwd, first, ModArith<FAST>{q},
        [&](uint32_t sub, uint32_t pos) {
            const uint64_t v = g[(size_t)pos * R2 + sub];
            return (FAST ? v : reduce_any(v, q, mu)) + hq;
        },
        [&](uint32_t sub, uint32_t pos, uint64_t v) { o[(size_t)pos * R2 + sub] = v; });
}

// forward, low stages, then y' = (y_l - t) * q_{Lc-1}^-1
template <int LOGN, bool FAST, int LP>
__global__ void __launch_bounds__(LowPassPolys<LOGN, LP>::threads, LP ? 3 : 12) k_fwd_low(Args A)
{
    using PS = LowPassPolys<LOGN, LP>;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t tile = blockIdx.x & ((1u << PS::ltiles) - 1), tr = blockIdx.x >> PS::ltiles;
    const uint32_t p0 = (tr / (A.Lc - 1)) << PS::lpolys, l = tr % (A.Lc - 1);
    const uint32_t first = tile << PS::lrows;
    const size_t so = (size_t)(A.Lc - 1) << LOGN, sy = (size_t)A.Lc << LOGN;
    const size_t at = ((size_t)l << LOGN) + ((size_t)first << PS::s);
    uint64_t *o = A.out + p0 * so + at;
    const uint64_t *y = A.polys + p0 * sy + at;
    const uint32_t np = A.count - p0;
    const NttLimb &Tl = A.T[l];
    const uint64_t q = Tl.q;
    const Twiddle qi = Tl.qinv[A.Lc - 1];
    // transform values: below 110q (FAST) or 12q; M = 128q or 12q bounds them
    const uint64_t M = (FAST ? 128 : 12) * q;
    constexpr int le = PS::s + PS::lrows;  // log2 elements per poly
    fwd_low_pass<LOGN, PS>(
        smem_raw, Tl.fwd, first, ModArith<FAST>{q}, np,
        [&] {
            // y is read only by the epilogue: start bringing it into L2 now
            for (uint32_t e = threadIdx.x * 16; e < PS::tile; e += PS::threads * 16)
                if ((e >> le) < np)
                    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(y + (e >> le) * sy + (e & ((1u << le) - 1))));
        },
        [&](uint32_t sub, uint32_t pos) {
            return o[(sub >> PS::lrows) * so + ((sub & (PS::rows - 1)) << PS::s) + pos];
        },
        [&](auto t_of) {
            sweep<PS, uint64_t>(
                np, [&](uint32_t e0, uint32_t t) { return y[(e0 >> le) * sy + (e0 & ((1u << le) - 1)) + t]; },
                [&](uint32_t e0, uint32_t t, uint64_t v) {
                    o[(e0 >> le) * so + (e0 & ((1u << le) - 1)) + t] =
                        canon6(mul_twiddle(v + M - t_of(e0, t), qi, q), q);
                });
        });
}

typedef void (*Kern)(Args);

// A ring dimension's launches; the low passes with one poly a CTA and with kPolys
struct Kernels {
    Kern inv_low[2], inv_high, fwd_high[2], fwd_low[2][2];
    // log2 tiles per transform, threads and shared memory per CTA
    uint32_t lt_low, lt_high, t_low[2], t_high;
    size_t s_low[2], s_high;
};

template <int LOGN>
constexpr Kernels kernels_for()
{
    typedef ModArith<false> MA;
    using Low1 = LowPassPolys<LOGN, 0>;
    using Low = LowPassPolys<LOGN>;
    using High = HighPass<LOGN>;
    static_assert((int)Low1::ltiles == (int)Low::ltiles, "the same tiles");
    return Kernels{{k_inv_low<LOGN, 0>, k_inv_low<LOGN, kLogPolys>},
                   k_inv_high<LOGN>,
                   {k_fwd_high<LOGN, false>, k_fwd_high<LOGN, true>},
                   {{k_fwd_low<LOGN, false, 0>, k_fwd_low<LOGN, false, kLogPolys>},
                    {k_fwd_low<LOGN, true, 0>, k_fwd_low<LOGN, true, kLogPolys>}},
                   Low::ltiles,
                   High::ltiles,
                   {Low1::threads, Low::threads},
                   High::threads,
                   {Low1::template smem_bytes<MA>(), Low::template smem_bytes<MA>()},
                   High::template smem_bytes<MA>()};
}

const Kernels &kernels(uint32_t n)
{
    static const Kernels K[] = {kernels_for<10>(), kernels_for<11>(), kernels_for<12>(), kernels_for<13>(),
                                kernels_for<14>(), kernels_for<15>(), kernels_for<16>(), kernels_for<17>()};
    return K[n - kLogNMin];
}

// ---------------------------------------------------------------------------
// Host: tables, built once per context on its first rescale
// ---------------------------------------------------------------------------
uint64_t mulm(uint64_t a, uint64_t b, uint64_t q) { return (uint64_t)((u128)a * b % q); }

uint64_t powm(uint64_t b, uint64_t e, uint64_t q)
{
    uint64_t r = 1 % q;
    b %= q;
    for (; e; e >>= 1) {
        if (e & 1) r = mulm(r, b, q);
        b = mulm(b, b, q);
    }
    return r;
}

// x * w mod q for a fixed w, with floor(2^64 w / q): no division a product
struct FixedMul {
    uint64_t w, wq, q;
    FixedMul(uint64_t w_, uint64_t q_) : w(w_), wq((uint64_t)(((u128)w_ << 64) / q_)), q(q_) {}
    uint64_t operator()(uint64_t x) const
    {
        const uint64_t r = x * w - (uint64_t)((u128)x * wq >> 64) * q;  // below 2q
        return r >= q ? r - q : r;
    }
};

// the table entry of w (ntt.cuh): 2^32 w mod q, and both quotients by 2q
Twiddle twiddle(uint64_t w, uint64_t q)
{
    const u128 w32 = (u128)w << 32;
    const uint64_t qw = (uint64_t)(w32 / q), v = (uint64_t)w32 - qw * q;
    Twiddle t;
    t.wv = make_ulonglong2(w, v);
    t.om = make_uint2((uint32_t)(qw / 2), (uint32_t)(((u128)v << 31) / q));
    return t;
}

// The least primitive 2N-th root of unity mod q, or 0.  For the first x whose
// c = x^((q-1)/2N) has c^N = -1, c is primitive and the primitive roots are
// its odd powers; the least of them is returned.
uint64_t least_root(uint64_t q, uint32_t N)
{
    const uint64_t M = 2ull * N;
    if ((q - 1) % M) return 0;
    uint64_t g = 0;
    for (uint64_t x = 2; x < 1000000 && x < q; ++x) {
        const uint64_t c = powm(x, (q - 1) / M, q);
        if (powm(c, N, q) == q - 1) {
            g = c;
            break;
        }
    }
    if (!g) return 0;
    const FixedMul by_g2(mulm(g, g, q), q);
    uint64_t best = g, cur = g;
    for (uint32_t j = 1; j < N; ++j) {
        cur = by_g2(cur);
        best = std::min(best, cur);
    }
    return best;
}

std::mutex g_ntt_mu;

int build_tables(const fiona_ctx *ctx)
{
    std::lock_guard<std::mutex> lock(g_ntt_mu);
    if (ctx->d_ntt) return FIONA_OK;
    const uint32_t N = ctx->N, L = ctx->L;
    // the shape of the low pass (LowPassPolys): n1 stages in the high pass,
    // tiles of 2^lrows rows
    const uint32_t n = log2u(N), n1 = n / 2, lrows = kLogTileMax - (n - n1) - kLogPolys;
    const size_t head = ((sizeof(NttLimb) * L + 255) / 256) * 256;
    const size_t wv = sizeof(ulonglong2) * N, om = sizeof(uint2) * N, table = wv + om, qtab = sizeof(Twiddle) * L;
    const size_t per_limb = 2 * table + ((qtab + 255) / 256) * 256;
    const size_t bytes = head + per_limb * L;
    std::vector<uint8_t> host(bytes, 0);
    std::vector<uint64_t> pw(N);
    void *dev = nullptr;
    cudaError_t e = cudaMalloc(&dev, bytes);
    if (e != cudaSuccess) return set_error(FIONA_ERR_NOMEM, "rescale tables: %s", cudaGetErrorString(e));
    for (uint32_t l = 0; l < L; ++l) {
        const uint64_t q = ctx->moduli[l];
        const uint64_t psi = least_root(q, N);
        if (!psi) {
            cudaFree(dev);
            return set_error(FIONA_ERR_MODULUS, "rescale: modulus %u has no primitive 2N-th root of unity", l);
        }
        const size_t off = head + per_limb * l;
        Twiddle *qinv = reinterpret_cast<Twiddle *>(host.data() + off + 2 * table);
        // powers of psi, then of psi^-1, placed in bit-reversed order
        for (int dir = 0; dir < 2; ++dir) {
            const uint64_t base = dir == 0 ? psi : powm(psi, q - 2, q);
            const FixedMul by_base(base, q);
            pw[0] = 1;
            for (uint32_t i = 1; i < N; ++i) pw[i] = by_base(pw[i - 1]);
            ulonglong2 *d_wv = reinterpret_cast<ulonglong2 *>(host.data() + off + dir * table);
            uint2 *d_om = reinterpret_cast<uint2 *>(host.data() + off + dir * table + wv);
            for (uint32_t k = 0; k < N; ++k) {
                const Twiddle t = twiddle(pw[bit_reverse(k, n)], q);
                const uint32_t at = low_place(k, n1, n - n1, lrows);
                d_wv[at] = t.wv;
                d_om[at] = t.om;
            }
        }
        for (uint32_t j = l + 1; j < L; ++j) qinv[j] = twiddle(powm(ctx->moduli[j] % q, q - 2, q), q);
        NttLimb &T = reinterpret_cast<NttLimb *>(host.data())[l];
        const uint8_t *dbase = static_cast<const uint8_t *>(dev) + off;
        T.fwd.wv = reinterpret_cast<const ulonglong2 *>(dbase);
        T.fwd.om = reinterpret_cast<const uint2 *>(dbase + wv);
        T.inv.wv = reinterpret_cast<const ulonglong2 *>(dbase + table);
        T.inv.om = reinterpret_cast<const uint2 *>(dbase + table + wv);
        T.qinv = reinterpret_cast<const Twiddle *>(dbase + 2 * table);
        T.q = q;
        T.mu64 = ~(uint64_t)0 / q;
        T.ninv = twiddle(powm(N % q, q - 2, q), q);
    }
    e = cudaMemcpy(dev, host.data(), bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(dev);
        return set_error(FIONA_ERR_CUDA, "rescale tables: %s", cudaGetErrorString(e));
    }
    ctx->d_ntt = dev;
    return FIONA_OK;
}

}  // namespace

int ntt_tables(const fiona_ctx *ctx, const fiona_ntt::NttLimb **limbs)
{
    const int rc = build_tables(ctx);
    if (rc == FIONA_OK) *limbs = reinterpret_cast<const NttLimb *>(ctx->d_ntt);
    return rc;
}

// One poly a CTA (64 threads) where those CTAs are few, up to `per_sm` an SM: a
// CTA of eight polys takes longer and leaves more of the GPU idle; and where the
// groups of eight are mostly absent polys, up to `few` of eight.  Both by the
// measured times: the one-poly CTAs of 2^7 and 2^8 positions idle half their
// threads in rounds of four stages.  GB300, rescale of 12 limbs, one poly against
// eight a CTA: 2^16, one poly 35.0 us against 44.3, two 47.3 - 50.4, three 56.5 -
// 53.6; 2^17, one 43.3 - 76.0, four 96.5 - 107.7, eight 171.5 - 163.2; 2^14, four
// 31.0 - 32.9, sixteen 53.4 - 49.4; 2^10, any count to 32 18.6 - 24.8.
bool many_polys(const fiona_ctx *ctx, uint64_t count, uint32_t limbs)
{
    const uint32_t n = log2u(ctx->N), s = n - n / 2;
    const uint64_t ctas = count * ((uint64_t)limbs << (n - kLogTileMax + kLogPolys));
    const uint64_t groups = (count + kPolys - 1) / kPolys;
    const uint64_t few = s == 8 ? 2 : s == 7 ? 4 : 5, per_sm = s == 8 ? 2 : s == 7 ? 5 : 13;
    return ctas > per_sm * std::max(ctx->sm_count, 1) && count > few * groups;
}

int launch_rescale(const fiona_ctx *ctx, void *stream, uint32_t Lc, uint64_t count, uint64_t *polys, uint64_t *out,
                   bool round)
{
    const NttLimb *T = nullptr;
    const int rc = ntt_tables(ctx, &T);
    if (rc) return rc;
    if (count == 0) return FIONA_OK;
    const uint32_t n = log2u(ctx->N);
    if (n < (uint32_t)kLogNMin || n > (uint32_t)kLogNMax)
        return set_error(FIONA_ERR_ARG, "rescale: N = %u outside [2^%d, 2^%d]", ctx->N, kLogNMin, kLogNMax);
    // the reduction-free forward butterflies need q < 2^56 and r < 4 q_l
    bool fast = true;
    const uint64_t qlast = ctx->moduli[Lc - 1];
    for (uint32_t l = 0; l + 1 < Lc; ++l)
        if (ctx->moduli[l] >= (1ull << 56) || qlast >= 4 * ctx->moduli[l]) fast = false;
    const Kernels &K = kernels(n);
    cudaError_t e = cudaSuccess;
    {
        // the dynamic shared memory limits, once per device and ring dimension
        static bool configured[FIONA_MAX_DEVICES][kLogNMax - kLogNMin + 1] = {};
        std::lock_guard<std::mutex> lock(g_ntt_mu);
        if (ctx->device < 0 || ctx->device >= FIONA_MAX_DEVICES)
            return set_error(FIONA_ERR_ARG, "rescale: device %d", ctx->device);
        if (!configured[ctx->device][n - kLogNMin]) {
            auto limit = [&](Kern k, size_t bytes) {
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute((const void *)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
            };
            limit(K.inv_high, K.s_high);
            for (int f = 0; f < 2; ++f) limit(K.fwd_high[f], K.s_high);
            for (int m = 0; m < 2; ++m) {
                limit(K.inv_low[m], K.s_low[m]);
                for (int f = 0; f < 2; ++f) limit(K.fwd_low[f][m], K.s_low[m]);
            }
            if (e != cudaSuccess)
                return set_error(FIONA_ERR_CUDA, "rescale: kernel attributes: %s", cudaGetErrorString(e));
            configured[ctx->device][n - kLogNMin] = true;
        }
    }
    // grid.x < 2^31: transforms * tiles, in chunks of whole polys
    const uint64_t max_polys = ((1ull << 31) - 1) / ((uint64_t)(Lc - 1) << std::max(K.lt_low, K.lt_high));
    cudaStream_t s = (cudaStream_t)stream;
    for (uint64_t p0 = 0; p0 < count && e == cudaSuccess; p0 += max_polys) {
        const uint64_t np = std::min<uint64_t>(count - p0, max_polys);
        Args a;
        a.polys = polys + p0 * Lc * (uint64_t)ctx->N;
        a.out = out + p0 * (Lc - 1) * (uint64_t)ctx->N;
        a.T = T;
        a.count = (uint32_t)np;
        a.Lc = Lc;
        a.round = round ? 1 : 0;
        const uint64_t nf = np * (Lc - 1);
        const int mi = many_polys(ctx, np, 1), mf = many_polys(ctx, np, Lc - 1);
        const uint64_t gi = mi ? (np + kPolys - 1) / kPolys : np, gf = mf ? (np + kPolys - 1) / kPolys : np;
        K.inv_low[mi]<<<(uint32_t)(gi << K.lt_low), K.t_low[mi], K.s_low[mi], s>>>(a);
        K.inv_high<<<(uint32_t)(np << K.lt_high), K.t_high, K.s_high, s>>>(a);
        K.fwd_high[fast]<<<(uint32_t)(nf << K.lt_high), K.t_high, K.s_high, s>>>(a);
        K.fwd_low[fast][mf]<<<(uint32_t)((gf * (Lc - 1)) << K.lt_low), K.t_low[mf], K.s_low[mf], s>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return set_error(FIONA_ERR_CUDA, "rescale launch: %s", cudaGetErrorString(e));
    return FIONA_OK;
}

void free_rescale_tables(const fiona_ctx *ctx)
{
    if (ctx->d_ntt) cudaFree(ctx->d_ntt);
    ctx->d_ntt = nullptr;
}
