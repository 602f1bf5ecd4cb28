"""Which kernel and shape a plan takes by itself (FIONA_KERNEL_AUTO), on both
sides of the rule's lines: the direct kernel where the model of its time is far
enough below the tiled kernel's, unless a shape of the tiled kernel is asked for;
the tiled kernel's shape where the model of its time moves it.  Every choice
gives the same residues (GPU parity)."""
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
    (112, 3, 3, 60, 0.9, True), (112, 4, 3, 60, 0.9, False),     # many inputs, few outputs
    (64, 1, 4, 50, 0.5, True),                                   # one output
])
def test_direct_kernel(n_in, n_out, L, bits, signed, direct):
    k = stats(n_in, n_out, L=L, bits=bits, signed=signed)["kernel"]
    assert k == (F.FIONA_KERNEL_DIRECT if direct else F.FIONA_KERNEL_TILED)


# at N = 2^12 and 3 limbs, the inputs up to which a layer of n outputs is direct:
# one group a term (a batch of four each on the tiled kernel), one group an output
SMALL = {(True, 50): {2: 7, 3: 9, 4: 13, 6: 21}, (False, 50): {3: 6, 4: 7, 6: 10, 8: 10, 12: 13, 16: 17},
         (False, 60): {2: 7, 3: 9, 4: 9, 6: 19, 8: 17, 12: 25}}


@pytest.mark.parametrize("per_term,bits,n_out", [(*k, n) for k, v in SMALL.items() for n in v])
def test_small_launches(per_term, bits, n_out):
    """One line in the inputs, direct below it and tiled above, which moves up
    with the outputs, the modulus and the groups."""
    line = SMALL[per_term, bits][n_out]
    got = [stats(n_in, n_out, N=4096, L=3, bits=bits, per_term=per_term)["kernel"] == F.FIONA_KERNEL_DIRECT
           for n_in in (line // 2, max(line * 2 // 3, 2), line * 4 // 3 + 1, line * 2 + 2)]
    assert got == [True, True, False, False], got


@pytest.mark.parametrize("n_in,n_out,N,bits,few,many", [(16, 16, 2048, 50, 2, 6), (24, 24, 4096, 50, 1, 6),
                                                        (7, 7, 65536, 50, 2, 8), (11, 11, 65536, 60, 2, 8)])
def test_fewer_limbs(n_in, n_out, N, bits, few, many):
    """The choice goes by the limbs of a launch: direct for few of them."""
    assert stats(n_in, n_out, N=N, L=few, bits=bits)["kernel"] == F.FIONA_KERNEL_DIRECT
    assert stats(n_in, n_out, N=N, L=many, bits=bits)["kernel"] == F.FIONA_KERNEL_TILED


@pytest.mark.parametrize("n_in,n_out,N,L,signed,matrix", [
    (96, 96, 1 << 16, 12, 0.53, True), (80, 17, 1 << 15, 2, 0.9, True),
    (12, 91, 1 << 15, 2, 0.5, True), (12, 91, 1 << 15, 1, 0.5, True), (12, 91, 1 << 11, 1, 0.5, False),
    (16, 10, 1 << 14, 2, 0.0, False), (19, 11, 1 << 15, 6, 0.3, False), (8, 8, 1 << 16, 12, 0.5, False),
])
def test_matrix_kernel(n_in, n_out, N, L, signed, matrix):
    """Constant raw plaintexts: the matrix kernel (128 coefficients a unit) where
    its time leads those of both others."""
    tern = int(n_in * n_out * signed)
    desc = W.constant_raw_plan(W.dense_hybrid_plan(W.PlanRng(7), n_in, n_out, tern // 2, tern // 2, 0))
    assert (stats(0, 0, N=N, L=L, desc=desc)["tile_coeffs"] == 128) == matrix


def test_smallest_layer_and_overrides(monkeypatch):
    wl = W.make_workload("tiny")
    assert stats(8, 4, N=wl.N, L=wl.L, bits=40, desc=wl.plan)["kernel"] == F.FIONA_KERNEL_DIRECT
    monkeypatch.setenv("FIONA_TILED_SHAPE", "2,4,1")
    assert stats(6, 6, N=4096, L=3)["kernel"] == F.FIONA_KERNEL_TILED


def test_tiled_shape():
    """Two coefficients per lane with one source region, where two regions fit
    only with one; the shapes of the measured layers as they were."""
    assert stats(100, 40, N=1 << 15, L=8, signed=0.6)["tile_coeffs"] == 64
    assert stats(125, 52, N=1 << 15, L=8, bits=60, signed=1.0)["tile_coeffs"] == 64
    for name, coeffs, warps in (("vgg", 32, 16), ("vit", 64, 8), ("bert", 64, 12)):
        wl = W.make_workload(name)
        s = stats(0, 0, N=wl.N, L=wl.L, desc=wl.plan)
        assert (s["tile_coeffs"], s["warps_per_cta"]) == (coeffs, warps)
