// encode.cu -- plaintext encoding on the GPU (Sec. 2.2 "Ciphertexts and
// Slots": CKKS packs a vector of numbers into the slots of a plaintext; the
// evaluated layer's gamma and raw plaintexts are such encodings of the
// model's weights, and the paper's timings include encoding them).
//
// Encoding of a slot vector z (N/2 complex numbers) at scale Delta:
//   1. embedding: m is the real poly of degree < N with m(zeta^(5^j)) = z_j
//      and m(zeta^(-5^j)) = conj(z_j), zeta = exp(i pi / N) (slot j sits at
//      the odd power 5^j mod 2N; the powers +-5^j are every odd residue);
//      the integer coefficients are c_i = round(Delta * m_i), ties away from
//      zero.  By the inversion formula over the odd powers of zeta,
//      m_i = (2/N) Re(u_i) and m_{i+n} = (2/N) Im(u_i), n = N/2, with
//        u_i = sum_j z_j zeta^(-5^j i) = sum_r y_r zeta^(-(4r+1) i),
//      y_r = z_j for 5^j = 4r + 1 mod 2N (the powers of 5 are the residues
//      1 mod 4), so
//        u_i = zeta^-i sum_r y_r omega^(r i),  omega = exp(-2 pi i / n),
//      a cyclic transform of size n = R1 R2.  The low pass gathers y in
//      bit-reversed order, transforms rows of R2 (row p holds the r = brv(p)
//      mod R1), and multiplies element (p, c) by omega^(brv(p) c) zeta^-c; the
//      high pass transforms the columns (R1 elements each) and, since zeta^-i
//      = zeta^-c zeta^(-R2 q) for i = R2 q + c, multiplies by Delta (2/N)
//      zeta^(-R2 q) and rounds the real and imaginary parts to the 64-bit
//      coefficients i and i + n.
//      The fp64 pipe bounds it (2 lanes a cycle and SM): about 50 fp64
//      operations a slot at 2^15 slots (a butterfly six, or four additions
//      where the twiddle is 1 or -i) against 66 with the negacyclic
//      Gentleman-Sande stages before, whose butterflies take eight.  Measured
//      on GB300, 93 vectors of 2^15 slots: 0.435 -> 0.326 ms.
//   2. RNS/NTT form: c_i mod q_l for every limb, then the forward NTT mod
//      q_l (ntt.cuh, the tables the rescale uses), canonical.
// Step 1 is floating point: it reproduces round(Delta m_i) except where
// Delta m_i lies within the transform's rounding error of a half-integer.
// Step 2 is exact.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "fiona_internal.h"
#include "ntt.cuh"

using namespace fiona_ntt;

namespace {

// in device memory, complex numbers as (cos, sin)
struct EncTables {
    const double2 *tw;       // [R2]: exp(-i pi m / h) at h + m, m < h, h a power of two
    const double2 *mid;      // [n]: omega^(brv(p) c) zeta^-c at p R2 + c
    const double2 *twist;    // [R1]: zeta^(-R2 q)
    const uint32_t *gather;  // [n]: the slot of y_brv(k)
};

struct EmbArgs {
    const double2 *slots;  // [count][N/2]
    double2 *work;         // [count][N/2]
    int64_t *coeffs;       // [count][N]
    EncTables E;
    double factor;         // Delta (2 / N)
    int *err;              // bit 1: a coefficient reached 2^62 (or was not finite)
};

struct EncArgs {
    const int64_t *coeffs;  // [count][N]
    uint64_t *out;          // [count][Lc][N]
    const NttLimb *T;
    uint32_t count;
    uint32_t Lc;
};

// round(x) as a 64-bit integer; 0 and the range flag when |x| >= 2^62 or x
// is not finite
__device__ __forceinline__ int64_t round_coeff(double x, int *err)
{
    if (fabs(x) < 0x1p62) return llround(x);
    atomicOr(err, 2);
    return 0;
}

// embedding, rows of the size-n transform (LN = log2 n): y in bit-reversed
// order gathered from the slots
template <int LN>
__global__ void __launch_bounds__(LowPass<LN>::threads, 4) k_embed_low(EmbArgs A)
{
    using PS = LowPass<LN>;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t tile = blockIdx.x & ((1u << PS::ltiles) - 1), p = blockIdx.x >> PS::ltiles;
    const uint32_t first = tile << PS::lsubs;
    const size_t base = (size_t)first << PS::s;
    const double2 *z = A.slots + ((size_t)p << LN);
    const uint32_t *gat = A.E.gather + base;
    const double2 *mid = A.E.mid + base;
    double2 *w = A.work + ((size_t)p << LN) + base;
    inv_low_pass<LN, PS>(
        smem_raw, A.E.tw, first, CplxArith{}, 1, [&](uint32_t e0, uint32_t t) { return z[gat[e0 + t]]; },
        [&](uint32_t sub, uint32_t pos, double2 v) {
            const uint32_t e = (sub << PS::s) + pos;
            w[e] = CplxArith::mul(v, mid[e]);
        });
}

// embedding, columns, then the last twist with Delta (2/N), rounded to the
// coefficients i and i + n
template <int LN>
__global__ void __launch_bounds__(HighPass<LN>::threads, 2) k_embed_high(EmbArgs A)
{
    using SH = Shape<LN>;
    using PS = HighPass<LN>;
    constexpr uint32_t R2 = 1u << (LN - SH::n1);
    extern __shared__ __align__(16) uint8_t smem_raw[];
    __shared__ double2 s_twist[1 << SH::n1];
    const uint32_t tile = blockIdx.x & ((1u << PS::ltiles) - 1), p = blockIdx.x >> PS::ltiles;
    const uint32_t first = tile << PS::lsubs;
    const double2 *g = A.work + ((size_t)p << LN) + first;
    int64_t *c = A.coeffs + ((size_t)p << (LN + 1)) + first;
    for (uint32_t q = threadIdx.x; q < (1u << SH::n1); q += PS::threads) {
        const double2 t = A.E.twist[q];
        s_twist[q] = make_double2(t.x * A.factor, t.y * A.factor);
    }
    __syncthreads();
    inv_high_pass<LN>(
        smem_raw, A.E.tw, first, CplxArith{}, [&](uint32_t sub, uint32_t pos) { return g[(size_t)pos * R2 + sub]; },
        [&](uint32_t sub, uint32_t pos, double2 v) {
            const size_t i = (size_t)pos * R2 + sub;
            const double2 u = CplxArith::mul(v, s_twist[pos]);
            c[i] = round_coeff(u.x, A.err);
            c[i + (1u << LN)] = round_coeff(u.y, A.err);
        });
}

// RNS/NTT form, forward high stages: c mod q_l into out (lazy)
template <int LOGN, bool FAST>
__global__ void __launch_bounds__(HighPass<LOGN>::threads, 3) k_enc_high(EncArgs A)
{
    using SH = Shape<LOGN>;
    using PS = HighPass<LOGN>;
    constexpr uint32_t R2 = 1u << (LOGN - SH::n1);
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t tile = blockIdx.x & ((1u << PS::ltiles) - 1), tr = blockIdx.x >> PS::ltiles;
    const uint32_t p = tr / A.Lc, l = tr % A.Lc;
    const uint32_t first = tile << PS::lsubs;
    const int64_t *c = A.coeffs + ((size_t)p << LOGN) + first;
    uint64_t *o = A.out + ((size_t)tr << LOGN) + first;
    const NttLimb &Tl = A.T[l];
    const uint64_t q = Tl.q, mu = Tl.mu64;
    fwd_high_pass<LOGN>(
        smem_raw, Tl.fwd, first, ModArith<FAST>{q},
        [&](uint32_t sub, uint32_t pos) {
            const int64_t v = c[(size_t)pos * R2 + sub];
            // the coefficients of a plaintext are mostly far below q: v + 4q
            // is then a value the reduction-free butterflies take, for two
            // additions and a comparison in place of a 64-bit high product
            // (GB300, 93 plaintexts of 2^16 at 12 limbs: 0.685 -> 0.631 ms)
            if (FAST && (uint64_t)v + 4 * q < 8 * q) return (uint64_t)v + 4 * q;
            // |v| as an unsigned word (exact for every 64-bit v); -|v| is q - r,
            // in (0, q]
            const uint64_t mag = v >= 0 ? (uint64_t)v : 0 - (uint64_t)v;
            const uint64_t r = reduce_any(mag, q, mu);
            return v >= 0 ? r : q - r;
        },
        [&](uint32_t sub, uint32_t pos, uint64_t v) { o[(size_t)pos * R2 + sub] = v; });
}

// RNS/NTT form, forward low stages, canonical store: the same rows of kPolys
// polys per CTA, or of one (many_polys; blockIdx.x = (group * Lc + limb) * tiles
// + tile)
template <int LOGN, bool FAST, int LP>
__global__ void __launch_bounds__(LowPassPolys<LOGN, LP>::threads, LP ? 4 : 12) k_enc_low(EncArgs A)
{
    using PS = LowPassPolys<LOGN, LP>;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t tile = blockIdx.x & ((1u << PS::ltiles) - 1), tr = blockIdx.x >> PS::ltiles;
    const uint32_t p0 = (tr / A.Lc) << PS::lpolys, l = tr % A.Lc;
    const uint32_t first = tile << PS::lrows;
    const size_t so = (size_t)A.Lc << LOGN;
    uint64_t *o = A.out + p0 * so + ((size_t)l << LOGN) + ((size_t)first << PS::s);
    const uint32_t np = A.count - p0;
    const NttLimb &Tl = A.T[l];
    const uint64_t q = Tl.q, mu = Tl.mu64;
    constexpr int le = PS::s + PS::lrows;  // log2 elements per poly
    fwd_low_pass<LOGN, PS>(
        smem_raw, Tl.fwd, first, ModArith<FAST>{q}, np, [] {},
        [&](uint32_t sub, uint32_t pos) {
            return o[(sub >> PS::lrows) * so + ((sub & (PS::rows - 1)) << PS::s) + pos];
        },
        [&](auto t_of) {
            sweep<PS, uint64_t>(
                np, [&](uint32_t e0, uint32_t t) { return t_of(e0, t); },
                [&](uint32_t e0, uint32_t t, uint64_t v) {
                    o[(e0 >> le) * so + (e0 & ((1u << le) - 1)) + t] = reduce_any(v, q, mu);
                });
        });
}

// ---------------------------------------------------------------------------
// Host
// ---------------------------------------------------------------------------
std::mutex g_enc_mu;

// exp(-i pi x / N) (host)
double2 unit_root(uint64_t x, uint32_t N)
{
    const long double a = -3.141592653589793238462643383279502884L * (long double)x / (long double)N;
    return make_double2((double)cosl(a), (double)sinl(a));
}

// byte offsets of the tables (n a power of two of at least 2^9: each part a
// multiple of 16 bytes)
struct EncOffsets {
    size_t tw = 0, mid, twist, gather, total;
    explicit EncOffsets(uint32_t n)
    {
        const uint32_t n1 = log2u(n) / 2;
        mid = tw + sizeof(double2) * (n >> n1);
        twist = mid + sizeof(double2) * n;
        gather = twist + (sizeof(double2) << n1);
        total = gather + sizeof(uint32_t) * n;
    }
};

int build_encode_tables(const fiona_ctx *ctx)
{
    std::lock_guard<std::mutex> lock(g_enc_mu);
    if (ctx->d_enc) return FIONA_OK;
    const uint32_t N = ctx->N, n = N / 2, ln = log2u(n), M = 2 * N;
    const uint32_t n1 = ln / 2, R1 = 1u << n1, R2 = n >> n1;
    const EncOffsets off(n);
    std::vector<uint8_t> host(off.total);
    double2 *tw = reinterpret_cast<double2 *>(host.data() + off.tw);
    double2 *mid = reinterpret_cast<double2 *>(host.data() + off.mid);
    double2 *twist = reinterpret_cast<double2 *>(host.data() + off.twist);
    uint32_t *gat = reinterpret_cast<uint32_t *>(host.data() + off.gather);
    auto unit = [=](uint64_t x) { return unit_root(x % M, N); };
    tw[0] = make_double2(1, 0);
    for (uint32_t h = 1; h < R2; h *= 2)
        for (uint32_t m = 0; m < h; ++m) tw[h + m] = unit((uint64_t)m * (N / h));
    for (uint32_t p = 0; p < R1; ++p)
        for (uint32_t c = 0; c < R2; ++c)  // omega = exp(-4 pi i / N)
            mid[p * R2 + c] = unit(4ull * bit_reverse(p, n1) * c + c);
    for (uint32_t q = 0; q < R1; ++q) twist[q] = unit((uint64_t)R2 * q);
    // slot j sits at the exponent 5^j mod 2N, which is 4r + 1 for one r < n
    std::vector<int64_t> slot_of_r(n, -1);
    uint64_t e5 = 1;
    for (uint32_t j = 0; j < n; ++j) {
        if (e5 % 4 != 1 || slot_of_r[(e5 - 1) / 4] >= 0)
            return set_error(FIONA_ERR_INTERNAL, "encode tables: 5^%u mod 2N = %llu", j, (unsigned long long)e5);
        slot_of_r[(e5 - 1) / 4] = j;
        e5 = e5 * 5 % M;
    }
    for (uint32_t k = 0; k < n; ++k) gat[k] = (uint32_t)slot_of_r[bit_reverse(k, ln)];
    void *dev = nullptr;
    cudaError_t err = cudaMalloc(&dev, off.total);
    if (err != cudaSuccess) return set_error(FIONA_ERR_NOMEM, "encode tables: %s", cudaGetErrorString(err));
    err = cudaMemcpy(dev, host.data(), off.total, cudaMemcpyHostToDevice);
    if (err != cudaSuccess) {
        cudaFree(dev);
        return set_error(FIONA_ERR_CUDA, "encode tables: %s", cudaGetErrorString(err));
    }
    ctx->d_enc = dev;
    return FIONA_OK;
}

typedef void (*EmbKern)(EmbArgs);
typedef void (*EncKern)(EncArgs);

template <int LOGN>
struct Inst {
    static constexpr size_t emb_low = LowPass<LOGN - 1>::template smem_bytes<CplxArith>();
    static constexpr size_t emb_high = HighPass<LOGN - 1>::template smem_bytes<CplxArith>();
    static constexpr size_t enc_low1 = LowPassPolys<LOGN, 0>::template smem_bytes<ModArith<false>>();
    static constexpr size_t enc_low = LowPassPolys<LOGN>::template smem_bytes<ModArith<false>>();
    static constexpr size_t enc_high = HighPass<LOGN>::template smem_bytes<ModArith<false>>();
};

struct Kernels {
    EmbKern emb_low, emb_high;
    EncKern enc_high[2], enc_low[2][2];  // by FAST; low pass: one poly a CTA, kPolys
    size_t s_emb_low, s_emb_high, s_enc_high, s_enc_low[2];
    // log2 tiles per transform and threads per CTA of each pass
    uint32_t lt_emb_low, lt_emb_high, lt_enc_high, lt_enc_low;
    uint32_t t_emb_low, t_emb_high, t_enc_high, t_enc_low[2];
};

template <int LOGN>
constexpr Kernels kernels_for()
{
    return Kernels{k_embed_low<LOGN - 1>,
                   k_embed_high<LOGN - 1>,
                   {k_enc_high<LOGN, false>, k_enc_high<LOGN, true>},
                   {{k_enc_low<LOGN, false, 0>, k_enc_low<LOGN, false, kLogPolys>},
                    {k_enc_low<LOGN, true, 0>, k_enc_low<LOGN, true, kLogPolys>}},
                   Inst<LOGN>::emb_low,
                   Inst<LOGN>::emb_high,
                   Inst<LOGN>::enc_high,
                   {Inst<LOGN>::enc_low1, Inst<LOGN>::enc_low},
                   LowPass<LOGN - 1>::ltiles,
                   HighPass<LOGN - 1>::ltiles,
                   HighPass<LOGN>::ltiles,
                   LowPassPolys<LOGN>::ltiles,
                   LowPass<LOGN - 1>::threads,
                   HighPass<LOGN - 1>::threads,
                   HighPass<LOGN>::threads,
                   {LowPassPolys<LOGN, 0>::threads, LowPassPolys<LOGN>::threads}};
}

const Kernels &kernels(uint32_t n)
{
    static const Kernels K[] = {kernels_for<10>(), kernels_for<11>(), kernels_for<12>(), kernels_for<13>(),
                                kernels_for<14>(), kernels_for<15>(), kernels_for<16>(), kernels_for<17>()};
    return K[n - kLogNMin];
}

// the dynamic shared memory limits, once per device and ring dimension
int configure(const fiona_ctx *ctx, uint32_t n)
{
    static bool done[FIONA_MAX_DEVICES][kLogNMax - kLogNMin + 1] = {};
    std::lock_guard<std::mutex> lock(g_enc_mu);
    if (ctx->device < 0 || ctx->device >= FIONA_MAX_DEVICES)
        return set_error(FIONA_ERR_ARG, "encode: device %d", ctx->device);
    if (done[ctx->device][n - kLogNMin]) return FIONA_OK;
    const Kernels &K = kernels(n);
    const std::pair<const void *, size_t> fs[] = {
        {(const void *)K.emb_low, K.s_emb_low},         {(const void *)K.emb_high, K.s_emb_high},
        {(const void *)K.enc_high[0], K.s_enc_high},    {(const void *)K.enc_high[1], K.s_enc_high},
        {(const void *)K.enc_low[0][0], K.s_enc_low[0]}, {(const void *)K.enc_low[1][0], K.s_enc_low[0]},
        {(const void *)K.enc_low[0][1], K.s_enc_low[1]}, {(const void *)K.enc_low[1][1], K.s_enc_low[1]}};
    for (const auto &f : fs) {
        const cudaError_t e = cudaFuncSetAttribute(f.first, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.second);
        if (e != cudaSuccess) return set_error(FIONA_ERR_CUDA, "encode: kernel attributes: %s", cudaGetErrorString(e));
    }
    done[ctx->device][n - kLogNMin] = true;
    return FIONA_OK;
}

}  // namespace

int launch_embed(const fiona_ctx *ctx, void *stream, uint64_t count, const double *slots, double scale,
                 int64_t *coeffs, double *work)
{
    const uint32_t n = log2u(ctx->N);
    if (n < (uint32_t)kLogNMin || n > (uint32_t)kLogNMax)
        return set_error(FIONA_ERR_ARG, "encode: N = %u outside [2^%d, 2^%d]", ctx->N, kLogNMin, kLogNMax);
    int rc = build_encode_tables(ctx);
    if (rc == FIONA_OK) rc = configure(ctx, n);
    if (rc) return rc;
    if (count == 0) return FIONA_OK;
    const Kernels &K = kernels(n);
    const uint8_t *tab = static_cast<const uint8_t *>(ctx->d_enc);
    EmbArgs a;
    const EncOffsets off(ctx->N / 2);
    a.E.tw = reinterpret_cast<const double2 *>(tab + off.tw);
    a.E.mid = reinterpret_cast<const double2 *>(tab + off.mid);
    a.E.twist = reinterpret_cast<const double2 *>(tab + off.twist);
    a.E.gather = reinterpret_cast<const uint32_t *>(tab + off.gather);
    a.factor = 2.0 * scale / (double)ctx->N;
    a.err = ctx->d_kerr;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaSuccess;
    const uint64_t max_polys = ((1ull << 31) - 1) >> std::max(K.lt_emb_low, K.lt_emb_high);
    for (uint64_t p0 = 0; p0 < count && e == cudaSuccess; p0 += max_polys) {
        const uint64_t np = std::min<uint64_t>(count - p0, max_polys);
        a.slots = reinterpret_cast<const double2 *>(slots) + p0 * (ctx->N / 2);
        a.work = reinterpret_cast<double2 *>(work) + p0 * (ctx->N / 2);
        a.coeffs = coeffs + p0 * ctx->N;
        K.emb_low<<<(uint32_t)(np << K.lt_emb_low), K.t_emb_low, K.s_emb_low, s>>>(a);
        K.emb_high<<<(uint32_t)(np << K.lt_emb_high), K.t_emb_high, K.s_emb_high, s>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return set_error(FIONA_ERR_CUDA, "encode launch: %s", cudaGetErrorString(e));
    return FIONA_OK;
}

int launch_encode_coeffs(const fiona_ctx *ctx, void *stream, uint32_t Lc, uint64_t count, const int64_t *coeffs,
                         uint64_t *out)
{
    const uint32_t n = log2u(ctx->N);
    if (n < (uint32_t)kLogNMin || n > (uint32_t)kLogNMax)
        return set_error(FIONA_ERR_ARG, "encode: N = %u outside [2^%d, 2^%d]", ctx->N, kLogNMin, kLogNMax);
    const NttLimb *T = nullptr;
    int rc = ntt_tables(ctx, &T);
    if (rc == FIONA_OK) rc = configure(ctx, n);
    if (rc) return rc;
    if (count == 0) return FIONA_OK;
    // the reduction-free butterflies need every q_l < 2^56 and inputs below 8 q_l,
    // as k_enc_high loads them
    bool fast = true;
    for (uint32_t l = 0; l < Lc; ++l)
        if (ctx->moduli[l] >= (1ull << 56)) fast = false;
    const Kernels &K = kernels(n);
    EncArgs a;
    a.T = T;
    a.Lc = Lc;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaSuccess;
    const uint64_t max_polys = ((1ull << 31) - 1) / ((uint64_t)Lc << std::max(K.lt_enc_high, K.lt_enc_low));
    for (uint64_t p0 = 0; p0 < count && e == cudaSuccess; p0 += max_polys) {
        const uint64_t np = std::min<uint64_t>(count - p0, max_polys);
        a.coeffs = coeffs + p0 * ctx->N;
        a.out = out + p0 * Lc * (uint64_t)ctx->N;
        a.count = (uint32_t)np;
        const int many = many_polys(ctx, np, Lc);
        const uint64_t nt = np * Lc, ng = many ? (np + kPolys - 1) / kPolys : np;
        K.enc_high[fast]<<<(uint32_t)(nt << K.lt_enc_high), K.t_enc_high, K.s_enc_high, s>>>(a);
        K.enc_low[fast][many]<<<(uint32_t)((ng * Lc) << K.lt_enc_low), K.t_enc_low[many], K.s_enc_low[many], s>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return set_error(FIONA_ERR_CUDA, "encode launch: %s", cudaGetErrorString(e));
    return FIONA_OK;
}

void free_encode_tables(const fiona_ctx *ctx)
{
    if (ctx->d_enc) cudaFree(ctx->d_enc);
    ctx->d_enc = nullptr;
}
