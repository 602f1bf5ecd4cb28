"""GPU parity of the matrix kernel (kernel_gemm.cu): layers whose raw
plaintexts are all constant, as exact products of digits on the tensor cores.
The bar is bit-exact equality with the CPU oracle.  FIONA_CONST_GEMM=1 takes
the kernel wherever it can run; the cases sit at its edges: inputs around the
multiples of 16 its contraction steps by, outputs around its groups of 16, its
blocks of 32 and its chunks, outputs with neither route, the most raw terms an
accumulator holds (64) with the largest digits, and moduli of 34 to 50 bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2609_35352_gb300 import build as B  # noqa: E402
from paper_2609_35352_gb300 import fiona as F  # noqa: E402
from paper_2609_35352_gb300 import workloads as W  # noqa: E402

from gpu_util import DeviceLayer, to_device, to_host  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


def layer(n_in, n_out, raw_share, seed, raw_most=64, signed=True):
    """Constant raw terms with probability raw_share (at most raw_most an
    output), signed terms with a zero now and then; every fifth output has no
    signed term, every seventh no raw one, every eleventh neither."""
    rng = np.random.default_rng(seed)
    per_output, n_raw, gout = [], 0, []
    for j in range(n_out):
        row, raws = [], 0
        for i in range(n_in):
            if j % 11 == 10:
                continue
            if j % 7 != 6 and raws < raw_most and rng.random() < raw_share:
                row.append((i, W.TERM_RAW_CONST, 0, n_raw, 0))
                n_raw += 1
                raws += 1
            elif signed and j % 5 != 4:
                row.append((i, W.TERM_TERNARY, int(rng.choice([-1, 0, 1], p=[0.45, 0.1, 0.45])), 0, len(gout)))
        if any(t[1] == W.TERM_TERNARY for t in row):
            gout.append(j)
        per_output.append(row)
    return W.build_plan(n_in, n_out, per_output, n_raw + len(gout), [n_raw + g for g in range(len(gout))], gout, [],
                        []), n_raw


def workload(plan, n_raw, N, bits, L, seed, fill="uniform"):
    return W.Workload("gemm", N, W.ntt_primes(N, bits, L), plan, seed, fill=fill, const_pts=n_raw)


@pytest.mark.parametrize("n_in,n_out,share,N,bits,L,fill", [
    (1, 2, 1.0, 1024, 50, 2, "uniform"),
    (15, 16, 0.5, 1024, 40, 3, "uniform"),
    (16, 17, 0.6, 2048, 50, 1, "uniform"),
    (17, 32, 0.5, 1024, 34, 2, "uniform"),
    (33, 33, 0.4, 1024, 45, 2, "uniform"),
    (64, 48, 1.0, 1024, 50, 2, "max"),
    (70, 40, 0.5, 1024, 50, 2, "uniform"),
    (96, 49, 0.9, 1024, 50, 2, "max"),
    (96, 96, 0.5, 4096, 50, 2, "uniform"),
    (81, 200, 0.5, 1024, 48, 1, "uniform"),
])
def test_matrix_kernel_parity(n_in, n_out, share, N, bits, L, fill, monkeypatch):
    monkeypatch.setenv("FIONA_CONST_GEMM", "1")
    plan, n_raw = layer(n_in, n_out, share, 31 * n_in + n_out)
    wl = workload(plan, n_raw, N, bits, L, 900 + n_in, fill)
    dl = DeviceLayer(wl)
    dl.plan.select_kernel("tiled")
    st = dl.plan.stats()
    assert st["tile_coeffs"] == 128 and st["const_raw_all"] == 1, st
    want = oracle.linear_eval(plan, wl.moduli, dl.X, dl.P)
    for _ in range(2):
        dl.run()
        mism = np.argwhere(dl.outputs() != want)
        assert mism.shape[0] == 0, "first mismatches (j, c, l, k): %s of %d" % (mism[:5].tolist(), mism.shape[0])
    assert dl.ctx.device_check() == F.FIONA_OK


@pytest.mark.parametrize("n_in,n_out,bits", [
    (17, 17, (50, 34, 45, 40)),       # one step and a half of 16 inputs, a block with one group
    (33, 49, (34, 50, 42, 50)),       # an odd number of steps, a last block with one group
    (81, 200, (49, 36, 50)),          # two chunks of outputs: 128 and 72
])
def test_matrix_kernel_walk(n_in, n_out, bits, monkeypatch):
    """Several units a CTA, whose ranges cross limbs (of moduli of different
    widths: the digits and biases are made again) and chunks (other outputs):
    every barrier's parity, the unit's coordinates and the next unit's
    prefetches, counted on from unit to unit."""
    monkeypatch.setenv("FIONA_CONST_GEMM", "1")
    N = 8192
    moduli = [W.ntt_primes(N, b, 1 + i)[i] for i, b in enumerate(bits)]
    plan, n_raw = layer(n_in, n_out, 0.5, 7 * n_in)
    wl = W.Workload("gemm", N, moduli, plan, 31 + n_in, const_pts=n_raw)
    dl = DeviceLayer(wl)
    dl.plan.select_kernel("tiled")
    assert dl.plan.stats()["tile_coeffs"] == 128
    units = (2 if n_out > 128 else 1) * len(moduli) * (N // 128) * 2
    assert units > 2 * torch.cuda.get_device_properties(0).multi_processor_count
    dl.run()
    want = oracle.linear_eval(plan, wl.moduli, dl.X, dl.P)
    mism = np.argwhere(dl.outputs() != want)
    assert mism.shape[0] == 0, "first mismatches (j, c, l, k): %s of %d" % (mism[:5].tolist(), mism.shape[0])
    assert dl.ctx.device_check() == F.FIONA_OK


def test_matrix_kernel_extreme_digits(monkeypatch):
    """Weights and residues around 0, q / 2 and the digit boundaries, whose
    centred digits are the largest; 64 raw terms in every output."""
    monkeypatch.setenv("FIONA_CONST_GEMM", "1")
    n_in, n_out, N, L = 64, 16, 1024, 2
    per_output = [[(i, W.TERM_RAW_CONST, 0, 64 * j + i, 0) for i in range(n_in)] for j in range(n_out)]
    plan = W.build_plan(n_in, n_out, per_output, 64 * n_out, [], [], [], [])
    wl = workload(plan, 64 * n_out, N, 50, L, 7)
    dl = DeviceLayer(wl)
    dl.plan.select_kernel("tiled")
    assert dl.plan.stats()["tile_coeffs"] == 128
    X, P = dl.X.copy(), dl.P.copy()
    for l, q in enumerate(wl.moduli):
        h = q // 2
        values = [0, 1, q - 1, h, h - 1, h + 1, h + 128, h - 128, h - 129, h + 127, (h + (1 << 47)) % q]
        values += [(h + s * v) % q for s in (1, -1) for v in (0x7F7F7F7F7F, 0x8080808080, 0x1FF7F7F7F7F7F, 1 << 48)]
        for k, v in enumerate(values):
            X[:, :, l, k] = v
        for j in range(n_out):
            P[64 * j:64 * j + 64, l, :] = values[j % len(values)]
    dl.d_in.copy_(to_device(X).view(-1).view(dl.d_in.shape))
    dl.d_pt.copy_(to_device(P).view(-1).view(dl.d_pt.shape))
    dl.run()
    assert np.array_equal(dl.outputs(), oracle.linear_eval(plan, wl.moduli, X, P))


def test_matrix_kernel_levels_and_choice(monkeypatch):
    """A lower level through the matrix kernel; and what does not take it: a
    plain raw term, 65 raw terms in an output, a second scale group, 51-bit
    moduli, FIONA_CONST_GEMM=0."""
    monkeypatch.setenv("FIONA_CONST_GEMM", "1")
    plan, n_raw = layer(24, 20, 0.5, 3)
    wl = workload(plan, n_raw, 1024, 50, 3, 5)
    ctx = F.Context(wl.N, wl.moduli, device=0)
    p = F.Plan(ctx, plan)
    p.select_kernel("tiled")
    X, P = wl.host_inputs(), wl.host_plaintexts()
    Xl, Pl = np.ascontiguousarray(X[:, :, :2]), np.ascontiguousarray(P[:, :2])
    d_out = torch.full((plan.n_out * 2 * 2 * wl.N,), -1, dtype=torch.int64, device="cuda")
    p.eval_level(2, to_device(Xl), to_device(Pl), d_out)
    torch.cuda.synchronize()
    got = to_host(d_out).reshape(plan.n_out, 2, 2, wl.N)
    assert np.array_equal(got, oracle.linear_eval(plan, wl.moduli[:2], Xl, Pl))

    def tile(pl, bits=50):
        c = F.Context(1024, W.ntt_primes(1024, bits, 2), device=0)
        q = F.Plan(c, pl)
        q.select_kernel("tiled")
        return q.stats()["tile_coeffs"]

    assert tile(plan) == 128 and tile(plan, 51) < 128
    one_raw = layer(24, 20, 0.5, 3)[0]
    one_raw.terms["kind"][np.nonzero(one_raw.terms["kind"] == W.TERM_RAW_CONST)[0][0]] = W.TERM_RAW
    assert tile(one_raw) < 128
    rows = [[(i, W.TERM_RAW_CONST, 0, i, 0) for i in range(65)], [(0, W.TERM_RAW_CONST, 0, 0, 0)]]
    assert tile(W.build_plan(65, 2, rows, 65, [], [], [], [])) < 128
    rows = [[(0, W.TERM_TERNARY, 1, 0, 0), (1, W.TERM_TERNARY, 1, 0, 1), (2, W.TERM_RAW_CONST, 0, 0, 0)], []]
    assert tile(W.build_plan(3, 2, rows, 3, [1, 2], [0, 0], [], [])) < 128
    monkeypatch.setenv("FIONA_CONST_GEMM", "0")
    assert tile(plan) < 128


@pytest.mark.parametrize("late", [1, 2])
def test_matrix_kernel_wait_runs_out(late, monkeypatch):
    """A test-only plan (FIONA_TEST_GEMM_TIMEOUT) with waits bounded at 2 ms and
    barriers that expect one arrival too many: those of the digits (1: the
    issuing warp's wait runs out) or that of the accumulators (2: the workers'
    wait does, and the issuing warp has multiplications to wait for).  The CTA
    stops and frees its tensor memory, fiona_device_check reports FIONA_ERR_TIMEOUT
    once, and the next evaluation on the same context is exact."""
    monkeypatch.setenv("FIONA_CONST_GEMM", "1")
    monkeypatch.setenv("FIONA_TEST_GEMM_TIMEOUT", str(late))
    plan, n_raw = layer(40, 33, 0.5, 11)
    wl = workload(plan, n_raw, 1024, 50, 2, 17)
    dl = DeviceLayer(wl)
    dl.plan.select_kernel("tiled")
    assert dl.plan.stats()["tile_coeffs"] == 128
    dl.run()
    torch.cuda.synchronize()
    assert dl.ctx.device_check() == F.FIONA_ERR_TIMEOUT
    assert dl.ctx.device_check() == F.FIONA_OK  # the flag was cleared
    monkeypatch.delenv("FIONA_TEST_GEMM_TIMEOUT")
    p = F.Plan(dl.ctx, plan)
    p.select_kernel("tiled")
    p.eval(dl.d_in, dl.d_pt, dl.d_out)
    assert np.array_equal(dl.outputs(), oracle.linear_eval(plan, wl.moduli, dl.X, dl.P))
    assert dl.ctx.device_check() == F.FIONA_OK
