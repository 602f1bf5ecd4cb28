"""Performance cases of the evaluator: what a program that uses it has it do,
through the public entry points (paper_2609_35352_gb300.fiona, the binding of
include/fiona.h), from the smallest layer, where a call is all latency, to the
30 GB layer that bench.py runs.

A case is one pass of one of four operations:

  layer          the hybrid linear layer y = sum gamma (sum +-A) + sum P A over
                 RNS ciphertexts, by one of its entry points: "eval" (device
                 buffers), "level" (fewer limbs than the context), "rescale"
                 (the layer followed by its rescale, at a level) and "host"
                 (inputs and outputs in pinned host memory)
  rescale        the rescale of a batch of polys, quotient rounded down or to
                 the nearest
  encode_coeffs  integer plaintexts to RNS NTT form
  embed          slot vectors to integer coefficients (fp64)

The context, the plan and the model's plaintexts are what such a program keeps
between calls; each state has fresh inputs, made from the seed.
"""
import math

import numpy as np
import torch

from paper_2609_35352_gb300 import fiona as F
from paper_2609_35352_gb300 import workloads as W

STREAM_INPUTS, STREAM_PLAINTEXTS, STREAM_POLYS = 1, 2, 9


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def _layer(name, N, L, bits, n_in, n_out, plus, minus, zero, plan_seed, dag=0.0, per_term=False, const=False,
           entry="eval", level=0, nearest=False):
    c = {"op": "layer", "N": N, "L": L, "bits": bits, "n_in": n_in, "n_out": n_out, "plus": plus, "minus": minus,
         "zero": zero, "plan_seed": plan_seed, "dag": dag, "per_term": per_term, "const": const, "entry": entry,
         "level": level or L, "nearest": nearest}
    return dict(c, name=name) if name else c


def listed():
    S = W.SEED_BASE
    return [
        # the smallest layer of the repository: one call is launch latency
        _layer("tiny", 1 << 12, 3, 40, 8, 4, 8, 8, 3, S + 0, per_term=True),
        # the weighted sum of 64 ciphertexts of the paper's motivation table:
        # one output, every input read once
        _layer("wsum-hybrid", 1 << 16, 24, 50, 64, 1, 16, 16, 0, S + 33),
        # a convolution layer: many rotated inputs, few outputs, mostly signed
        _layer("vgg", 1 << 16, 20, 50, 144, 16, 819, 819, 182, S + 2),
        # a transformer projection, and deep in a model: fewer limbs left and
        # the layer's rescale with it, as the next layer needs it
        _layer("vit", 1 << 16, 16, 50, 32, 24, 225, 225, 49, S + 3, dag=0.25),
        _layer("vit-level-rescale", 1 << 16, 16, 50, 32, 24, 225, 225, 49, S + 3, dag=0.25, entry="rescale", level=7,
               nearest=True),
        # the largest single layer: a feed-forward block with a full plaintext
        # per weight group, and with weights broadcast to every slot
        _layer("bert", 1 << 16, 12, 50, 96, 96, 2198, 2198, 488, S + 4, dag=0.30),
        _layer("bert-const", 1 << 16, 12, 50, 96, 96, 2198, 2198, 488, S + 4, dag=0.30, const=True),
        # an ordinary layer of ragged size on 60-bit primes (few, wide limbs:
        # SEAL's largest), and a mid-size layer called on host buffers
        _layer("wide-ragged", 1 << 15, 5, 60, 37, 11, 120, 130, 17, S + 77),
        _layer("host-mid", 1 << 14, 8, 50, 24, 16, 110, 110, 20, S + 78, entry="host"),
        # the rescale of the largest layer's outputs as a call of its own
        {"op": "rescale", "N": 1 << 16, "L": 12, "bits": 50, "count": 192, "nearest": False, "name": "rescale-bert"},
        # loading a model: its plaintexts encoded on the GPU, in the two steps
        # of the encoder (an odd batch of them each)
        {"op": "encode_coeffs", "N": 1 << 16, "L": 12, "bits": 50, "count": 93, "name": "encode-coeffs"},
        {"op": "embed", "N": 1 << 16, "count": 93, "scale_bits": 46, "name": "embed"},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _limit(N, limbs, polys, most):
    """The largest L (at least 2) with polys * L * N * 8 bytes below `most`."""
    return max(2, min(limbs, int(most / (polys * N * 8.0))))


def draw(rng):
    most = 8e9  # bytes of one state: the largest listed case has 30e9
    N = 1 << rng.randint(12, 16)
    bits = rng.choice((40, 45, 50, 50, 50, 54, 60))
    kind = rng.choices(("layer", "rescale", "encode_coeffs", "embed"), (7, 2, 1, 1))[0]
    if kind == "embed":
        return {"op": "embed", "N": N, "count": _log(rng, 1, 300), "scale_bits": rng.randint(36, 46)}
    if kind != "layer":
        count = _log(rng, 1, 256) if kind == "encode_coeffs" else 2 * _log(rng, 1, 100)
        L = _limit(N, _log(rng, 2, 24), 3 * count, most)
        c = {"op": kind, "N": N, "L": L, "bits": bits, "count": count}
        return dict(c, nearest=rng.random() < 0.5) if kind == "rescale" else c
    n_in, n_out = _log(rng, 3, 150), _log(rng, 1, 100)
    pairs = n_in * n_out
    tern = rng.choice((0.0, 0.5, 0.55, 0.75, 0.8, 1.0, rng.random())) * pairs
    zero = int(0.1 * tern)
    plus = int((tern - zero) / 2)
    minus = plus
    raw = pairs - zero - plus - minus
    # shared sums of four inputs need outputs to share them
    dag = 0.25 if n_out >= 8 and n_in >= 16 and plus >= 64 and rng.random() < 0.4 else 0.0
    L = _limit(N, _log(rng, 2, 24), 2 * n_in + 4 * n_out + raw + n_out, most)
    entry = rng.choice(("eval", "eval", "eval", "level", "rescale", "rescale"))
    level = L if entry == "eval" else rng.randint(2, L)
    return _layer("", N, L, bits, n_in, n_out, plus, minus, zero, rng.randrange(1 << 30), dag=dag,
                  const=rng.random() < 0.15, entry=entry, level=level, nearest=rng.random() < 0.5)


# ----------------------------------------------------------------------------
# what the program keeps, and its inputs
# ----------------------------------------------------------------------------
_contexts = {}  # one context per (N, moduli), kept as a program keeps its own


def _moduli(case):
    return W.ntt_primes(case["N"], case.get("bits", 50), case.get("L", 1))


def _context(case):
    key = (case["N"], case.get("bits", 50), case.get("L", 1))
    if key not in _contexts:
        if len(_contexts) >= 4:
            _contexts.clear()
        ctx = F.Context(case["N"], _moduli(case), device=torch.cuda.current_device())
        # the transform tables are built by the context's first use of them
        if case["op"] == "encode_coeffs" or case["op"] == "rescale" or case.get("entry") == "rescale":
            z = torch.zeros(case["N"], dtype=torch.int64, device="cuda")
            ctx.encode_coeffs(1, 1, z, torch.empty_like(z))
        if case["op"] == "embed":
            z = torch.zeros((3, case["N"]), dtype=torch.float64, device="cuda")
            ctx.ckks_embed(1, z[0], 1.0, z[1], z[2])
        torch.cuda.synchronize()
        _contexts[key] = ctx
    return _contexts[key]


def _plan(case):
    p = W.dense_hybrid_plan(W.PlanRng(case["plan_seed"]), case["n_in"], case["n_out"], case["plus"], case["minus"],
                            case["zero"], group_per_term=case["per_term"], dag_share=case["dag"])
    return W.constant_raw_plan(p) if case["const"] else p


def _residues(outer, case, seed, stream, mode=0, limbs=None):
    """[outer][limbs][N] uniform residues on the GPU (mode 2: constant per limb)."""
    qs = _moduli(case)[: limbs or case["L"]]
    t = torch.empty((outer, len(qs), case["N"]), dtype=torch.int64, device="cuda")
    if outer:
        F.device_fill(t, outer, len(qs), case["N"], qs, W.stream_key(seed, stream), mode)
    return t


def _inputs(case, seed):
    """The GPU tensors a pass reads, from the case and the seed alone."""
    if case["op"] == "layer":
        p, lv = _plan(case), case["level"]
        x = _residues(2 * p.n_in, case, seed, STREAM_INPUTS, limbs=lv)
        pt = _residues(p.n_pt, case, seed, STREAM_PLAINTEXTS, limbs=lv)
        raw = p.counts()["raw"]
        if case["const"] and raw:  # the raw plaintexts come first
            F.device_fill(pt, raw, lv, case["N"], _moduli(case)[:lv], W.stream_key(seed, STREAM_PLAINTEXTS), 2)
        return p, x.view(p.n_in, 2, lv, case["N"]), pt
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["op"] == "rescale":
        return _residues(case["count"], case, seed, STREAM_POLYS)
    if case["op"] == "encode_coeffs":
        # encoded weights at scale 2^46: coefficients of a few times 2^40
        return torch.randn((case["count"], case["N"]), generator=g, device="cuda", dtype=torch.float64).mul_(
            2.0 ** 41).round_().to(torch.int64)
    z = torch.randn((case["count"], case["N"] // 2, 2), generator=g, device="cuda", dtype=torch.float64) * 0.1
    z[..., 1] = 0  # model weights are real
    return z


def prepare(case, seed):
    ctx = _context(case)
    s = {"case": case, "ctx": ctx}
    N = case["N"]

    def empty(*shape):
        return torch.empty(shape, dtype=torch.int64, device="cuda")

    if case["op"] == "layer":
        desc, x, pt = _inputs(case, seed)
        lv = case["level"]
        s.update(plan=F.Plan(ctx, desc), x=x, pt=pt, out=empty(desc.n_out, 2, lv, N))
        if case["entry"] == "rescale":
            s["rescaled"] = empty(desc.n_out, 2, lv - 1, N)
        if case["entry"] == "host":
            s["h_in"] = x.cpu().pin_memory()
            s["h_out"] = torch.empty(s["out"].shape, dtype=torch.int64).pin_memory()
    elif case["op"] == "rescale":
        s.update(x=_inputs(case, seed), out=empty(case["count"], case["L"] - 1, N))
    elif case["op"] == "encode_coeffs":
        s.update(x=_inputs(case, seed), out=empty(case["count"], case["L"], N))
    else:
        s.update(x=_inputs(case, seed), out=empty(case["count"], N),
                 work=torch.empty((case["count"], N), dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    return s


def run(s):
    case, stream = s["case"], torch.cuda.current_stream()
    if case["op"] == "rescale":
        # leaves the coefficients of each poly's last limb in the input
        s["ctx"].rescale(case["L"], case["count"], s["x"], s["out"], stream=stream, round=case["nearest"])
        return s["out"]
    if case["op"] == "encode_coeffs":
        s["ctx"].encode_coeffs(case["L"], case["count"], s["x"], s["out"], stream=stream)
        return s["out"]
    if case["op"] == "embed":
        s["ctx"].ckks_embed(case["count"], s["x"], 2.0 ** case["scale_bits"], s["out"], s["work"], stream=stream)
        return s["out"]
    plan = s["plan"]
    if case["entry"] == "eval":
        plan.eval(s["x"], s["pt"], s["out"], stream=stream)
        return s["out"]
    if case["entry"] == "level":
        plan.eval_level(case["level"], s["x"], s["pt"], s["out"], stream=stream)
        return s["out"]
    if case["entry"] == "rescale":
        plan.eval_rescale(case["level"], s["x"], s["pt"], s["out"], s["rescaled"], stream=stream,
                          round=case["nearest"])
        return s["rescaled"]
    plan.eval_host(s["h_in"], s["pt"], s["h_out"], s["x"], s["out"], stream=stream)
    return s["h_out"]


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def work(case):
    """bytes: each input residue read once, each output residue written once;
    flops: a multiply and an add per product of residues (or of doubles)."""
    N = case["N"]
    n = N.bit_length() - 1
    if case["op"] == "layer":
        p, lv = _plan(case), case["level"]
        groups = len(set(int(g) for g in p.terms["group"][(p.terms["kind"] == W.TERM_TERNARY) & (p.terms["sign"] != 0)]))
        prod = 2.0 * lv * N * (p.counts()["raw"] + groups)
        b = W.min_bytes(p, lv, N)
        if case["entry"] == "rescale":  # the layer's own outputs need not be kept
            b -= 2 * p.n_out * N * 8
            prod += 2.0 * p.n_out * (lv * N * n / 2 + (lv - 1) * N)
        return {"bytes": b, "flops": 2 * prod}
    if case["op"] == "embed":
        return {"bytes": case["count"] * N * 16, "flops": case["count"] * 10.0 * (N / 4) * (n - 1)}
    L, c = case["L"], case["count"]
    if case["op"] == "rescale":
        return {"bytes": c * (2 * L - 1) * N * 8, "flops": 2.0 * c * (L * N * n / 2 + (L - 1) * N)}
    return {"bytes": c * (L + 1) * N * 8, "flops": 2.0 * c * L * N * n / 2}


def tolerance(case):
    """Residues are elements of Z_q: whole numbers with one right value.  The
    embedding rounds fp64 sums to integers: another order of the transform
    moves a value near a half-integer to the next one (measured against
    exact() on the GB300: 1.4e-5 of the coefficients, by one)."""
    return {"differ": 6e-5} if case["op"] == "embed" else "exact"


# ----------------------------------------------------------------------------
# the same values in plain torch (64-bit integers, fp64 quotients)
# ----------------------------------------------------------------------------
def _mul30(a, b, q):
    """a * b mod q for 0 <= a < q < 2^60 and 0 <= b < 2^30: the quotient in fp64
    is at most a few off, and the remainder is taken modulo 2^64."""
    k = torch.floor(a.to(torch.float64) * b.to(torch.float64) / q.to(torch.float64)).to(torch.int64)
    return torch.remainder(a * b - k * q, q)


def _mul(a, b, q):
    """a * b mod q, b below 2^60 in two digits of 30 bits."""
    hi = _mul30(_mul30(a, b >> 30, q), torch.full_like(q, 1 << 30), q)
    return torch.remainder(hi + _mul30(a, b & ((1 << 30) - 1), q), q)


def _exact_layer(case, seed):
    p, x, pt = _inputs(case, seed)
    q = torch.tensor(_moduli(case)[: case["level"]], dtype=torch.int64, device="cuda").view(1, -1, 1)
    out = torch.zeros((p.n_out, 2, case["level"], case["N"]), dtype=torch.int64, device="cuda")
    for j in range(p.n_out):
        y = out[j]
        sums = {}
        for t in p.output_terms(j):
            i, kind, sign = int(t["input"]), int(t["kind"]), int(t["sign"])
            if kind == W.TERM_TERNARY:
                if sign:
                    g = int(t["group"])
                    s = sums.get(g)
                    v = x[i] if sign > 0 else q - x[i]
                    sums[g] = v if s is None else torch.remainder(s + v, q)
            else:
                w = pt[int(t["pt"])]
                if kind == W.TERM_RAW_CONST:
                    w = w[:, :1]
                y.copy_(torch.remainder(y + _mul(x[i], w.expand(x[i].shape), q), q))
        for g, s in sums.items():
            y.copy_(torch.remainder(y + _mul(s, pt[int(p.group_scale_pt[g])].expand(s.shape), q), q))
    return out


def _psi_powers(q, N, inverse):
    """psi^brv(k) (or psi^-brv(k)), k < N, psi the least primitive 2N-th root mod q."""
    n = N.bit_length() - 1
    g = next(c for c in (pow(x, (q - 1) // (2 * N), q) for x in range(2, 1000)) if pow(c, N, q) == q - 1)
    qt = torch.tensor([q], dtype=torch.int64, device="cuda")

    def powers(b, count):
        v = torch.ones(1, dtype=torch.int64, device="cuda")
        step = b
        while v.numel() < count:
            v = torch.cat((v, _mul(v, torch.full_like(v, step), qt)))
            step = step * step % q
        return v

    odd = _mul(powers(g * g % q, N), torch.full((N,), g, dtype=torch.int64, device="cuda"), qt)
    psi = int(odd.min())
    k = torch.arange(N, device="cuda")
    brv = torch.zeros_like(k)
    for b in range(n):
        brv |= ((k >> b) & 1) << (n - 1 - b)
    return powers(pow(psi, q - 2, q) if inverse else psi, N)[brv]


def _transform(a, q, N, inverse):
    """The negacyclic transform of the last axis ([..., N]) mod q, or its inverse."""
    w = _psi_powers(q, N, inverse)
    qt = torch.tensor(q, dtype=torch.int64, device="cuda")
    shape = a.shape
    sizes = [1 << s for s in range(N.bit_length() - 1)]
    for m in (reversed(sizes) if inverse else sizes):
        v = a.view(-1, m, 2, N // (2 * m))
        t = w[m:2 * m].view(1, m, 1)
        if inverse:
            hi = _mul(torch.remainder(v[:, :, 0] - v[:, :, 1], qt), t.expand(v[:, :, 0].shape), qt)
            lo = torch.remainder(v[:, :, 0] + v[:, :, 1], qt)
        else:
            u = _mul(v[:, :, 1], t.expand(v[:, :, 1].shape), qt)
            lo, hi = torch.remainder(v[:, :, 0] + u, qt), torch.remainder(v[:, :, 0] - u, qt)
        a = torch.stack((lo, hi), 2).reshape(shape)
    if inverse:
        a = _mul(a, torch.full_like(a, pow(N, q - 2, q)), qt)
    return a


def _exact_rescale(polys, qs, N, nearest):
    """[count][L][N] -> [count][L - 1][N]."""
    ql = qs[-1]
    r = _transform(polys[:, -1].contiguous(), ql, N, True)
    if nearest:
        r = torch.remainder(r + ql // 2, torch.tensor(ql, device="cuda"))
    out = torch.empty((polys.shape[0], len(qs) - 1, N), dtype=torch.int64, device="cuda")
    for l, q in enumerate(qs[:-1]):
        qt = torch.tensor(q, dtype=torch.int64, device="cuda")
        t = _transform(torch.remainder(r - (ql // 2 if nearest else 0), qt), q, N, False)
        d = torch.remainder(polys[:, l] - t, qt)
        out[:, l] = _mul(d, torch.full_like(d, pow(ql, q - 2, q)), qt)
    return out


def exact(case, seed):
    N = case["N"]
    if case["op"] == "layer":
        y = _exact_layer(case, seed)
        if case["entry"] == "rescale":
            lv = case["level"]
            y = _exact_rescale(y.view(-1, lv, N), _moduli(case)[:lv], N, case["nearest"]).view(-1, 2, lv - 1, N)
        return y.cpu() if case["entry"] == "host" else y
    if case["op"] == "rescale":
        return _exact_rescale(_inputs(case, seed), _moduli(case), N, case["nearest"])
    x = _inputs(case, seed)
    if case["op"] == "encode_coeffs":
        qs = _moduli(case)
        return torch.stack([_transform(torch.remainder(x, torch.tensor(q, device="cuda")), q, N, False) for q in qs], 1)
    # embed: slot j sits at zeta^(5^j); the exponents 4r + 1 in order of r
    n = N // 2
    e5 = np.empty(n, dtype=np.int64)
    e = 1
    for j in range(n):
        e5[(e - 1) // 4] = j
        e = e * 5 % (2 * N)
    y = torch.view_as_complex(x.contiguous())[:, torch.from_numpy(e5).cuda()]
    i = torch.arange(n, device="cuda", dtype=torch.float64) * (math.pi / N)
    u = torch.fft.fft(y, dim=1) * torch.polar(torch.ones_like(i), -i)
    m = torch.cat((u.real, u.imag), 1) * (2.0 * 2.0 ** case["scale_bits"] / N)
    return (torch.sign(m) * torch.floor(m.abs() + 0.5)).to(torch.int64)
