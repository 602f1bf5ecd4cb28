// lower_gemm.cpp -- lowering of a layer whose raw plaintexts are all constant
// to the matrix kernel's schedule (gemm.h), and the model of that kernel's time.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <set>

#include "gemm.h"

int gemm_configure(size_t smem);  // kernel_gemm.cu

namespace {

// the most dynamic shared memory a CTA may have (227 KB)
constexpr size_t kSmemMax = 232448;

}  // namespace

// Predicted SM cycles of a launch over `n_limbs` limbs: the making of G's digits,
// and the units of the CTA that has most, each by its blocks of 32 outputs,
// groups of 16 and inputs (fitted on GB300 to 1455 random layers of 2 to 96
// inputs and 2 to 100 outputs, N = 2^10 to 2^16, 1 to 12 limbs, 10 us to 2 ms, to
// the scale of the other kernels' models: 4% from the measured time, one standard
// deviation)
double gemm_cycles(const fiona_plan *p, uint32_t n_limbs)
{
    const GemmArgs &a = p->gemm->args;
    const uint32_t units = gemm_units(p, n_limbs), sms = p->ctx->sm_count > 0 ? p->ctx->sm_count : 152;
    const double chunks = a.n_chunks, groups = (a.n_out + 15) / 16 / chunks;
    const double blocks = (a.n_out + kGemmBlock - 1) / kGemmBlock / chunks;
    const double unit = 2130 + 1700 * blocks + (2450 + 12.4 * a.K) * groups + 47.0 * a.K;
    return 16400 + 9.5 * p->stats.n_raw_terms / chunks + (units + sms - 1) / sms * unit;
}

// Builds p->gemm where the matrix kernel can run the layer; leaves it null
// otherwise.  FIONA_CONST_GEMM=0 never builds it; =1 has it run whatever its time.
int lower_gemm(fiona_plan *p)
{
    const HostPlan &hp = p->hp;
    const fiona_ctx *ctx = p->ctx;
    const char *env = getenv("FIONA_CONST_GEMM");
    const bool off = env && env[0] == '0', force = env && env[0] == '1';
    // a forced shape of the tiled kernel is a request for that kernel
    if (off || (!force && p->shape_asked)) return FIONA_OK;
    if (!hp.n_in || hp.n_in > kGemmMaxInputs || hp.n_out < 2 || ctx->q_max >= (1ull << 50)) return FIONA_OK;
    for (const uint64_t q : ctx->moduli)
        if (q < (1ull << 33)) return FIONA_OK;
    // one entry per (output, input) and route, one scale group per output
    std::vector<GemmTerm> raw, sgn;
    std::vector<uint32_t> gamma(hp.n_out, kGemmNoGamma), raw_row(1, 0), sgn_row(1, 0);
    std::set<uint32_t> groups;
    for (uint32_t j = 0; j < hp.n_out; ++j) {
        std::set<uint32_t> in_raw, in_sgn;
        uint32_t group = 0;
        for (uint32_t e = hp.term_offsets[j]; e < hp.term_offsets[j + 1]; ++e) {
            const fiona_term &t = hp.terms[e];
            if (t.kind == FIONA_TERM_RAW) return FIONA_OK;
            if (t.kind == FIONA_TERM_RAW_CONST) {
                if (!in_raw.insert(t.input).second) return FIONA_OK;
                raw.push_back({0, (uint16_t)t.input, t.pt});
            } else if (t.sign != 0) {
                if (!in_sgn.insert(t.input).second) return FIONA_OK;
                if (gamma[j] != kGemmNoGamma && group != t.group) return FIONA_OK;
                group = t.group;
                groups.insert(group);
                gamma[j] = hp.group_scale_pt[t.group];
                sgn.push_back({0, (uint16_t)t.input, t.sign > 0 ? 1u : 0u});
            }
        }
        if (in_raw.size() > kGemmMaxRaw) return FIONA_OK;
        raw_row.push_back((uint32_t)raw.size());
        sgn_row.push_back((uint32_t)sgn.size());
    }
    if (raw.empty()) return FIONA_OK;

    const uint32_t K = (hp.n_in + 15) & ~15u, blocks = (hp.n_out + kGemmBlock - 1) / kGemmBlock;
    uint32_t fit = blocks;  // blocks of outputs per CTA
    const size_t cap = (ctx->smem_optin ? std::min(kSmemMax, ctx->smem_optin) : kSmemMax) - 256;  // (static words)
    while (fit && GemmLayout(K, fit * kGemmBlock).total > cap) --fit;
    if (!fit) return FIONA_OK;
    // (the outputs' biases are made by one worker each)
    fit = std::min(fit, kGemmEpilogueWarps * 32 / kGemmBlock);
    const uint32_t n_chunks = (blocks + fit - 1) / fit;
    const uint32_t chunk = (blocks + n_chunks - 1) / n_chunks * kGemmBlock;

    GemmSchedule *g = new GemmSchedule;
    g->smem = GemmLayout(K, chunk).total;
    g->groups = (uint32_t)groups.size();
    g->always = force;
    GemmArgs &a = g->args;
    a.limbs = ctx->d_limbs;
    a.err = ctx->d_kerr;
    a.N = ctx->N;
    a.n_in = hp.n_in;
    a.K = K;
    a.n_out = hp.n_out;
    a.chunk = chunk;
    a.n_chunks = n_chunks;
    a.wait_ns = 2000000000ull;
    if (const char *t = getenv("FIONA_TEST_GEMM_TIMEOUT")) {  // test only: a wait that runs out
        a.test_flags = (uint32_t)atoi(t) & (kGemmTestDigits | kGemmTestFull);
        if (a.test_flags) a.wait_ns = 2000000ull;
    }
    a.c1 = 1;
    a.c8 = 1u << 8;
    a.c16 = 1u << 16;
    a.c24 = 1u << 24;
    p->gemm = g;
    if (ctx->device == FIONA_DEVICE_NONE) return FIONA_OK;

    std::vector<uint32_t> raw_off, sgn_off;
    for (uint32_t c = 0; c <= n_chunks; ++c) {
        const uint32_t j = std::min(c * chunk, hp.n_out);
        raw_off.push_back(raw_row[j]);
        sgn_off.push_back(sgn_row[j]);
    }
    for (uint32_t j = 0; j < hp.n_out; ++j) {
        for (uint32_t e = raw_row[j]; e < raw_row[j + 1]; ++e) raw[e].out = (uint16_t)(j % chunk);
        for (uint32_t e = sgn_row[j]; e < sgn_row[j + 1]; ++e) sgn[e].out = (uint16_t)(j % chunk);
    }
    std::vector<uint8_t> blob;
    auto put = [&](const void *src, size_t bytes) {
        const size_t at = (blob.size() + 15) & ~(size_t)15;
        blob.resize(at + bytes);
        if (bytes) memcpy(blob.data() + at, src, bytes);
        return at;
    };
    const size_t o_raw = put(raw.data(), raw.size() * sizeof(GemmTerm));
    const size_t o_sgn = put(sgn.data(), sgn.size() * sizeof(GemmTerm));
    const size_t o_ro = put(raw_off.data(), raw_off.size() * 4), o_so = put(sgn_off.data(), sgn_off.size() * 4);
    const size_t o_g = put(gamma.data(), gamma.size() * 4);
    cudaError_t e = cudaMalloc(&g->sched.blob, blob.size());
    if (e != cudaSuccess) return set_error(FIONA_ERR_NOMEM, "matrix kernel schedule: %s", cudaGetErrorString(e));
    g->sched.bytes = blob.size();
    e = cudaMemcpy(g->sched.blob, blob.data(), blob.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return set_error(FIONA_ERR_CUDA, "matrix kernel schedule: %s", cudaGetErrorString(e));
    const uint8_t *d = static_cast<const uint8_t *>(g->sched.blob);
    a.raw = reinterpret_cast<const GemmTerm *>(d + o_raw);
    a.sgn = reinterpret_cast<const GemmTerm *>(d + o_sgn);
    a.raw_off = reinterpret_cast<const uint32_t *>(d + o_ro);
    a.sgn_off = reinterpret_cast<const uint32_t *>(d + o_so);
    a.gamma = reinterpret_cast<const uint32_t *>(d + o_g);
    return gemm_configure(g->smem);
}

void free_gemm(fiona_plan *p)
{
    if (!p->gemm) return;
    if (p->gemm->sched.blob) cudaFree(p->gemm->sched.blob);
    delete p->gemm;
    p->gemm = nullptr;
}
