"""Which kernel a plan takes by itself (FIONA_KERNEL_AUTO), around the lines of
the rule: outputs of few operands run on the direct kernel, unless a shape of
the tiled kernel is asked for.  Both give the same residues (GPU parity)."""
import pytest

from paper_2609_35352_gb300 import build as B
from paper_2609_35352_gb300 import fiona as F
from paper_2609_35352_gb300 import workloads as W


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def kernel(n_in, n_out, N=1 << 16, L=4, bits=50, per_term=False, desc=None):
    tern = n_in * n_out // 2
    desc = desc or W.dense_hybrid_plan(W.PlanRng(7), n_in, n_out, tern // 2, tern // 2, 0, group_per_term=per_term)
    ctx = F.Context(N, W.ntt_primes(N, bits, L), device=F.FIONA_DEVICE_NONE)
    return F.Plan(ctx, desc).stats()["kernel"]


@pytest.mark.parametrize("n_in,n_out,bits,direct", [
    (6, 6, 50, True), (7, 6, 50, False), (3, 54, 50, True),   # six operands an output
    (10, 10, 60, True), (11, 10, 60, False), (10, 10, 50, False),  # ten with wide moduli
    (16, 2, 50, True), (17, 2, 50, False),                    # two outputs
    (64, 1, 50, True),                                        # one
])
def test_few_operands(n_in, n_out, bits, direct):
    assert kernel(n_in, n_out, bits=bits) == (F.FIONA_KERNEL_DIRECT if direct else F.FIONA_KERNEL_TILED)


def test_size_groups_and_overrides(monkeypatch):
    assert kernel(8, 8, N=4096, L=2, bits=60) == F.FIONA_KERNEL_TILED  # wide, but too small a launch
    assert kernel(8, 4, per_term=True) == F.FIONA_KERNEL_DIRECT       # a batch of four per one-term group
    assert kernel(8, 4) == F.FIONA_KERNEL_TILED
    wl = W.make_workload("tiny")
    assert kernel(8, 4, N=wl.N, L=wl.L, bits=40, desc=wl.plan) == F.FIONA_KERNEL_DIRECT
    monkeypatch.setenv("FIONA_TILED_SHAPE", "2,4,1")
    assert kernel(6, 6) == F.FIONA_KERNEL_TILED
