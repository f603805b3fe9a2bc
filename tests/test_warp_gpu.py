"""Few output blocks on the CUDA cores run a warp per block, many the lane groups
(FP64) or register tiles (FP32) (GPU).  Every element is the same chain of
operations in either, so the first block rows of a product computed alone (few)
must be the bits of those rows in the whole product (many); the whole product
against the oracle, the adjoints of the few against the oracle's."""
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


def _first_rows(X, r):
    nnz = int(X.row_ptr[r])
    end = int(X.blk_off[nnz]) if nnz < X.nnzb else len(X.data)
    return I.BCSR(X.row_bs[:r], X.col_bs, X.row_ptr[:r + 1], X.col_idx[:nnz], X.blk_off[:nnz], X.data[:end])


SHAPES = [(3,), (4,), (5,), (6,), (8,), (13,), (17,), (28,), (33,), (4, 1), (5, 13, 23), (3, 7, 16, 32)]


@pytest.mark.parametrize("dtype", [np.float64, np.float32], ids=["fp64", "fp32"])
@pytest.mark.parametrize("sizes", SHAPES, ids=lambda s: "_".join(map(str, s)))
def test_few_and_many_agree(bsm, oracle, sizes, dtype):
    import torch
    nb = 400                                    # up to 160,000 blocks; the first 12 rows hold 4,800
    bs = I.mixed_sizes(nb, sizes, [1.0 / len(sizes)] * len(sizes), seed=5)
    Ah, Bh = random_bcsr(bs, bs, 0.1, seed=21, dtype=dtype), random_bcsr(bs, bs, 0.1, seed=22, dtype=dtype)
    C0 = random_bcsr(bs, bs, 0.2, seed=23, dtype=dtype)
    As, Cs = _first_rows(Ah, 12), _first_rows(C0, 12)
    B = bsm.Matrix.from_host(Bh)
    for flush in (0, 4):
        many = bsm.multiply(-0.75, bsm.Matrix.from_host(Ah), B, 0.5, bsm.Matrix.from_host(C0), 0.5, flush_every=flush)
        few = bsm.multiply(-0.75, bsm.Matrix.from_host(As), B, 0.5, bsm.Matrix.from_host(Cs), 0.5, flush_every=flush)
        part = few.data_host()
        np.testing.assert_array_equal(part, many.data_host()[:len(part)])
        if dtype == np.float64 and flush == 0:
            ref = oracle.multiply(-0.75, Ah, Bh, eps=0.5, beta=0.5, Cold=C0).C
            np.testing.assert_array_equal(many.pattern()[1], ref.col_idx)
            assert rel_fro(many.data_host(), ref.data) <= 1e-12
    if dtype == np.float64:                     # few blocks of A and of B: the adjoints' kernel as well
        A = bsm.Matrix.from_host(As)
        C = bsm.multiply(1.0, A, B)
        ref = oracle.multiply(1.0, As, Bh)
        G = np.linspace(-1.0, 1.0, ref.C.data_len)
        dA, dB = (torch.full((len(X.data),), np.nan, dtype=torch.float64, device="cuda") for X in (As, Bh))
        bsm.multiply_backward(0.5, C, torch.tensor(G, device="cuda"), A, B, dA, dB)
        for got, want in zip((dA, dB), oracle.multiply_backward(0.5, As, Bh, ref.C, G, ref.prods)):
            assert rel_fro(got.cpu().numpy(), want) <= 1e-12
