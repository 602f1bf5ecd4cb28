"""Plans that live side by side on one device: creating one leaves the others as
they were.  The dynamic shared memory a kernel may be launched with is a setting
of the kernel, which plans of different sizes share: a large plan evaluates, bit
for bit as the oracle, after a small one was created.  And one plan at every
level, whose launches differ in kernel."""
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


def layer(n_in, n_out, const):
    tern = n_in * n_out // 2
    p = W.dense_hybrid_plan(W.PlanRng(5), n_in, n_out, tern // 2, tern // 2, 0)
    if const:
        p = W.constant_raw_plan(p)
    wl = W.Workload("live", 1024, W.ntt_primes(1024, 50, 2), p, 3, const_pts=p.counts()["raw"] if const else 0)
    dl = DeviceLayer(wl)
    dl.plan.select_kernel("tiled")
    return dl


@pytest.mark.parametrize("env,const", [
    ({"FIONA_CONST_GEMM": "1"}, True),           # the matrix kernel
    ({"FIONA_TILED_SHAPE": "2,8,0"}, False),     # the tiled kernel, the same shape for both
    ({"FIONA_TILED_WS": "1", "FIONA_WS_SHAPE": "8,1,3"}, False),  # its warp-specialised variant
])
def test_large_plan_after_small(env, const, monkeypatch):
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    large, small = layer(96, 40, const), layer(20, 20, const)
    a, b = large.plan.stats(), small.plan.stats()
    assert a["kernel"] == b["kernel"] == F.FIONA_KERNEL_TILED and a["tile_coeffs"] == b["tile_coeffs"]
    assert a["smem_bytes"] > b["smem_bytes"] and a["smem_bytes"] > 48 * 1024
    for dl in (small, large, small):
        dl.run()
        assert np.array_equal(dl.outputs(), oracle.linear_eval(dl.wl.plan, dl.wl.moduli, dl.X, dl.P))


def test_every_level_of_one_plan():
    """The kernel goes by a launch's limbs: here the direct one up to 3 of 6, the
    tiled one for 4 and 6; both read buffers laid out for the level."""
    tern = 16 * 16 // 2
    p = W.dense_hybrid_plan(W.PlanRng(7), 16, 16, tern // 2, tern // 2, 0)
    wl = W.Workload("levels", 2048, W.ntt_primes(2048, 50, 6), p, 4)
    ctx = F.Context(wl.N, wl.moduli, device=0)
    plan = F.Plan(ctx, p)
    X, P = wl.host_inputs(), wl.host_plaintexts()
    for lv in range(1, 7):
        Xl, Pl = np.ascontiguousarray(X[:, :, :lv]), np.ascontiguousarray(P[:, :lv])
        out = torch.full((p.n_out * 2 * lv * wl.N,), -1, dtype=torch.int64, device="cuda")
        plan.eval_level(lv, to_device(Xl), to_device(Pl), out)
        torch.cuda.synchronize()
        got = to_host(out).reshape(p.n_out, 2, lv, wl.N)
        assert np.array_equal(got, oracle.linear_eval(p, wl.moduli[:lv], Xl, Pl)), lv
    assert ctx.device_check() == F.FIONA_OK
