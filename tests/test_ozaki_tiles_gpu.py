"""Half tiles of the Ozaki path (GPU): where at most 8 rows of an output block fall
into its last tile row, or at most 8 terms of k into a product's last step, only
the registers in use are packed, copied and multiplied.  Sizes on both sides of
every edge, in all three dimensions.  Integer data whose sums stay below 2^53 is
exact on this path, so those values must be equal; random data keeps the path's
1e-13 against the oracle."""
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


@pytest.mark.parametrize("inner", [(1, 8, 9), (16, 17, 24), (25, 32, 40)], ids=str)
@pytest.mark.parametrize("heights", [(6, 8, 9), (16, 17, 24), (25, 33, 41)], ids=str)
def test_sizes(bsm, oracle, heights, inner):
    rows = I.mixed_sizes(36, heights, [1 / 3] * 3, seed=3)
    mid = I.mixed_sizes(36, inner, [1 / 3] * 3, seed=4)
    cols = I.mixed_sizes(36, (7, 16, 23), [1 / 3] * 3, seed=5)
    Ah, Bh = random_bcsr(rows, mid, 0.3, seed=6), random_bcsr(mid, cols, 0.3, seed=7)
    for integers in (False, True):
        if integers:
            rng = np.random.default_rng(8)
            Ah.data[:] = rng.integers(-200, 201, len(Ah.data))
            Bh.data[:] = rng.integers(-200, 201, len(Bh.data))
        A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)
        C = bsm.multiply(1.0, A, B, prec="ozaki")
        ref = oracle.multiply(1.0, Ah, Bh)
        G = np.linspace(-1.0, 1.0, ref.C.data_len)
        if integers:
            G = np.round(150 * G)
        import torch
        dA = torch.full((len(Ah.data),), np.nan, dtype=torch.float64, device="cuda")
        dB = torch.full((len(Bh.data),), np.nan, dtype=torch.float64, device="cuda")
        bsm.multiply_backward(1.0, C, torch.from_numpy(G).cuda(), A, B, dA, dB, prec="ozaki")
        dA_ref, dB_ref = oracle.multiply_backward(1.0, Ah, Bh, ref.C, G, ref.prods)
        for got, want in ((C.data_host(), ref.C.data), (dA.cpu().numpy(), dA_ref), (dB.cpu().numpy(), dB_ref)):
            if integers:
                np.testing.assert_array_equal(got, want)
            else:
                assert rel_fro(got, want) <= 1e-13


@pytest.mark.parametrize("nb,occ", [(60, 0.08), (60, 0.5), (150, 0.3), (250, 0.13)],
                         ids=["whole", "half", "half_many", "whole_many"])
@pytest.mark.parametrize("heights", [(23,), (5, 13, 23), (17, 40, 6)], ids=str)
@pytest.mark.parametrize("band", [False, True], ids=["uniform", "band"])
def test_whole_and_half_layouts(bsm, oracle, band, heights, nb, occ):
    """Below five products a block the operands are packed in whole tiles, else in half ones where they end in half a
    tile; a band has more products a block than the uniform pattern that the first guess assumes.  Small integers:
    exact either way, forward, adjoints and a no-sync call with other values."""
    import torch
    rows = I.mixed_sizes(nb, heights, [1 / len(heights)] * len(heights), seed=3)
    mid = I.mixed_sizes(nb, (5, 16, 24), [1 / 3] * 3, seed=4)
    rng = np.random.default_rng(8)
    if band:                       # the same number of blocks, in a band twice as wide as full
        near = [(i, j) for i in range(nb) for j in range(nb) if abs(i - j) <= nb * occ]
        Ah, Bh = (I.assemble(x, y, *np.array([p for p in near if rng.random() < 0.5]).T, None, seed=s)
                  for x, y, s in ((rows, mid, 6), (mid, rows, 7)))
    else:
        Ah, Bh = random_bcsr(rows, mid, occ, seed=6), random_bcsr(mid, rows, occ, seed=7)
    for X in (Ah, Bh):
        X.data[:] = rng.integers(-8, 9, len(X.data))
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)
    C = bsm.multiply(1.0, A, B, prec="ozaki")
    ref = oracle.multiply(1.0, Ah, Bh)
    np.testing.assert_array_equal(C.pattern()[1], ref.C.col_idx)
    np.testing.assert_array_equal(C.data_host(), ref.C.data)
    G = rng.integers(-8, 9, ref.C.data_len).astype(np.float64)
    dA, dB = (torch.full((len(X.data),), np.nan, dtype=torch.float64, device="cuda") for X in (Ah, Bh))
    bsm.multiply_backward(1.0, C, torch.tensor(G, device="cuda"), A, B, dA, dB, prec="ozaki")
    for got, want in zip((dA, dB), oracle.multiply_backward(1.0, Ah, Bh, ref.C, G, ref.prods)):
        np.testing.assert_array_equal(got.cpu().numpy(), want)
    Ah.data[:] = rng.integers(-8, 9, len(Ah.data))
    A.set_data(Ah.data)
    bsm.multiply(1.0, A, B, Cm=C, prec="ozaki", no_sync=True)
    np.testing.assert_array_equal(C.data_host(), oracle.multiply(1.0, Ah, Bh).C.data)
