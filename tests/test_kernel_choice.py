"""Which kernel and shape a plan takes by itself (FIONA_KERNEL_AUTO), on both
sides of the rule's lines: the direct kernel where the model of its time is a
tenth below the tiled kernel's, and for small launches of few operands an
output, unless a shape of the tiled kernel is asked for; the tiled kernel's shape
where the model of its time moves it.  Every choice gives the same residues (GPU
parity)."""
import pytest

from paper_2609_35352_gb300 import build as B
from paper_2609_35352_gb300 import fiona as F
from paper_2609_35352_gb300 import workloads as W


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def stats(n_in, n_out, N=1 << 16, L=4, bits=50, signed=0.5, per_term=False, desc=None):
    tern = int(n_in * n_out * signed)
    desc = desc or W.dense_hybrid_plan(W.PlanRng(7), n_in, n_out, tern // 2, tern // 2, 0, group_per_term=per_term)
    ctx = F.Context(N, W.ntt_primes(N, bits, L), device=F.FIONA_DEVICE_NONE)
    return F.Plan(ctx, desc).stats()


@pytest.mark.parametrize("n_in,n_out,L,bits,signed,direct", [
    (3, 49, 4, 60, 0.54, True), (3, 73, 10, 40, 0.0, False),     # three operands an output: wide, narrow
    (4, 9, 13, 45, 0.95, True), (6, 65, 2, 50, 0.1, False),
    (113, 9, 5, 60, 1.0, True), (112, 4, 3, 60, 0.9, False),     # many inputs, few outputs
    (64, 1, 4, 50, 0.5, True),                                   # one output
])
def test_direct_kernel(n_in, n_out, L, bits, signed, direct):
    k = stats(n_in, n_out, L=L, bits=bits, signed=signed)["kernel"]
    assert k == (F.FIONA_KERNEL_DIRECT if direct else F.FIONA_KERNEL_TILED)


def test_small_launches_and_overrides(monkeypatch):
    small = dict(N=4096, L=3)
    assert stats(6, 6, **small)["kernel"] == F.FIONA_KERNEL_DIRECT    # six operands an output
    assert stats(7, 6, **small)["kernel"] == F.FIONA_KERNEL_TILED
    assert stats(4, 2, **small)["kernel"] == F.FIONA_KERNEL_TILED     # two outputs
    assert stats(8, 4, **small)["kernel"] == F.FIONA_KERNEL_TILED
    wl = W.make_workload("tiny")  # a batch of four per one-term group
    assert stats(8, 4, N=wl.N, L=wl.L, bits=40, desc=wl.plan)["kernel"] == F.FIONA_KERNEL_DIRECT
    monkeypatch.setenv("FIONA_TILED_SHAPE", "2,4,1")
    assert stats(6, 6, **small)["kernel"] == F.FIONA_KERNEL_TILED


def test_tiled_shape():
    """Two coefficients per lane with one source region, where two regions fit
    only with one; the shapes of the measured layers as they were."""
    assert stats(100, 40, N=1 << 15, L=8, signed=0.6)["tile_coeffs"] == 64
    assert stats(125, 52, N=1 << 15, L=8, bits=60, signed=1.0)["tile_coeffs"] == 64
    for name, coeffs, warps in (("vgg", 32, 16), ("vit", 64, 8), ("bert", 64, 12)):
        wl = W.make_workload(name)
        s = stats(0, 0, N=wl.N, L=wl.L, desc=wl.plan)
        assert (s["tile_coeffs"], s["warps_per_cta"]) == (coeffs, warps)
