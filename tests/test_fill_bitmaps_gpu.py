"""The fill's two ways of building a C block's products (GPU): common bits of
A's row and B's column where the filter can drop nothing of the row, a walk of
B's column elsewhere.  Patterns, product lists and values against the oracle
with thresholds on both sides of the switch, inner dimensions around a bitmap
word and around the 32 words a warp expands at a time, and norms that are NaN,
infinite and zero (the oracle's rule: kept only if the product exceeds eps)."""
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


def _check(bsm, oracle, Ah, Bh, eps, beta=0.0, C0=None):
    Cm = None if C0 is None else bsm.Matrix.from_host(C0)
    C = bsm.multiply(1.0, bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh), beta, Cm, eps)
    ref = oracle.multiply(1.0, Ah, Bh, eps=eps, beta=beta, Cold=C0)
    rp, ci, bo = C.pattern()
    np.testing.assert_array_equal(rp, ref.C.row_ptr)
    np.testing.assert_array_equal(ci, ref.C.col_idx)
    np.testing.assert_array_equal(bo, ref.C.blk_off)
    p = C.products()
    for x, y in ((p.a, ref.prods.a), (p.b, ref.prods.b), (p.c, ref.prods.c)):
        np.testing.assert_array_equal(x, y)
    return C.data_host(), ref.C.data


@pytest.mark.parametrize("nbk", [1, 31, 32, 33, 1023, 1024, 1025, 1500])
def test_inner_dimensions(bsm, oracle, nbk):
    rows, cols, inner = I.uniform_sizes(20, 2), I.uniform_sizes(37, 3), I.mixed_sizes(nbk, (1, 2), (0.5, 0.5), seed=3)
    Ah, Bh = random_bcsr(rows, inner, 0.4, seed=81), random_bcsr(inner, cols, 0.4, seed=82)
    for eps in (0.0, 1e-12, 1.0):
        c, ref = _check(bsm, oracle, Ah, Bh, eps)
        assert rel_fro(c, ref) <= 1e-12


def test_threshold_at_the_smallest_product(bsm, oracle):
    bs = I.uniform_sizes(60, 4)
    Ah, Bh = random_bcsr(bs, bs, 0.3, seed=83), random_bcsr(bs, bs, 0.3, seed=84)
    C0 = random_bcsr(bs, bs, 0.1, seed=85)
    least = bsm.Matrix.from_host(Ah).block_norms().min() * bsm.Matrix.from_host(Bh).block_norms().min()
    for eps in (np.nextafter(least, 0.0), least, np.nextafter(least, 9.0), 3.0 * least):
        c, ref = _check(bsm, oracle, Ah, Bh, float(eps), -0.5, C0)
        assert rel_fro(c, ref) <= 1e-12


def test_norms_that_are_not_finite(bsm, oracle):
    bs = I.uniform_sizes(40, 2)
    Ah, Bh = random_bcsr(bs, bs, 0.3, seed=86), random_bcsr(bs, bs, 0.3, seed=87)
    Ah.data[0], Ah.data[40], Bh.data[8], Bh.data[80] = np.nan, np.inf, np.inf, np.nan
    Ah.data[100:104] = 0.0
    _check(bsm, oracle, Ah, Bh, 1e-9)
    Bh.data[80] = 1.0   # no NaN in B: only A's rows with one walk
    _check(bsm, oracle, Ah, Bh, 1e-9)
