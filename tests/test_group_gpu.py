"""The FP64 kernel's lane groups (GPU): output blocks of every layout the
kernel chooses from (a warp per block, several blocks per warp in row- or
column-keeping groups, several passes over large blocks), with enough blocks
that small ones share a warp.  Every element is one chain of FP64 fused
multiply-adds in ascending k whatever the layout, so the builds (which choose
different layouts) must agree bit for bit; against the oracle 1e-12."""
import numpy as np
import pytest

from paper_1708_03604_gb300 import inputs as I
from tests.helpers import random_bcsr, rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bsm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_03604_gb300 import bsm as B
    B.lib()
    return B


def _with_builds(bsm, call):
    """call() under every build the kernel may be asked for; the results must be the same bits."""
    from paper_1708_03604_gb300 import autotune
    got = []
    try:
        for build in (-1, 1, 2):
            bsm.bsm_set_tuning("fp64", "fp64_build", build)
            got.append(call())
    finally:
        autotune.reset("fp64")
    for g in got[1:]:
        for x, y in zip(got[0], g):
            np.testing.assert_array_equal(x, y)
    return got[0]


SHAPES = [(1,), (2,), (3,), (4,), (5,), (6,), (8,), (9,), (13,), (17,), (28,), (4, 1), (5, 13, 23), (3, 7, 16, 32)]


@pytest.mark.parametrize("sizes", SHAPES, ids=lambda s: "_".join(map(str, s)))
def test_layouts_agree_and_match_oracle(bsm, oracle, sizes):
    import torch
    nb = 170 if max(sizes) < 28 else 100
    bs = I.mixed_sizes(nb, sizes, [1.0 / len(sizes)] * len(sizes), seed=5)
    # a few rows of A hold nothing: C blocks there come from the old C alone
    Ah, Bh = random_bcsr(bs, bs, 0.12, seed=21), random_bcsr(bs, bs, 0.12, seed=22)
    C0 = random_bcsr(bs, bs, 0.2, seed=23)
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)

    def plain():
        C = bsm.multiply(1.0, A, B)
        g = torch.linspace(-1.0, 1.0, C.info().data_len, dtype=torch.float64, device="cuda")
        dA = torch.full((len(Ah.data),), np.nan, dtype=torch.float64, device="cuda")
        dB = torch.full((len(Bh.data),), np.nan, dtype=torch.float64, device="cuda")
        bsm.multiply_backward(0.5, C, g, A, B, dA, dB)
        return C.data_host(), dA.cpu().numpy(), dB.cpu().numpy()

    c, dA, dB = _with_builds(bsm, plain)
    ref = oracle.multiply(1.0, Ah, Bh)
    assert rel_fro(c, ref.C.data) <= 1e-12
    G = np.linspace(-1.0, 1.0, ref.C.data_len)
    dA_ref, dB_ref = oracle.multiply_backward(0.5, Ah, Bh, ref.C, G, ref.prods)
    assert rel_fro(dA, dA_ref) <= 1e-12 and rel_fro(dB, dB_ref) <= 1e-12

    def merged():
        return (bsm.multiply(-0.75, A, B, 0.5, bsm.Matrix.from_host(C0), 0.9).data_host(),)

    c, = _with_builds(bsm, merged)
    ref = oracle.multiply(-0.75, Ah, Bh, eps=0.9, beta=0.5, Cold=C0)
    assert rel_fro(c, ref.C.data) <= 1e-12


def test_non_finite_values_stay_in_their_rows(bsm):
    """Infinities and NaN reach exactly the elements whose chain holds them (idle lane slots read no other block)."""
    bs = I.uniform_sizes(150, 5)
    Ah, Bh = random_bcsr(bs, bs, 0.1, seed=31), random_bcsr(bs, bs, 0.1, seed=32)
    base = bsm.multiply(1.0, bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)).to_host()
    Ah.data[7], Ah.data[1003] = np.inf, np.nan
    got = bsm.multiply(1.0, bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)).to_host()
    brow = np.repeat(np.arange(150), np.diff(Ah.row_ptr))
    bad = {(int(brow[e // 25]), (e % 25) // 5) for e in (7, 1003)}
    crow = np.repeat(np.arange(150), np.diff(got.row_ptr))
    rows = np.stack([np.repeat(crow, 25), np.tile(np.arange(25) // 5, len(crow))], 1)
    hit = np.array([(int(i), int(r)) in bad for i, r in rows])
    np.testing.assert_array_equal(got.data[~hit], base.data[~hit])
    assert not np.isfinite(got.data[hit]).all()
