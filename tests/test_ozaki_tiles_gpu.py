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
