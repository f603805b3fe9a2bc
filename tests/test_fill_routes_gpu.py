"""Which way the fill builds C's products (GPU): bitmaps of B's columns where the
columns are long for the inner dimension and the products many, a walk of the
columns elsewhere and where the bitmaps' memory is refused.  The route shows in
the allocations of the multiply; patterns, product lists and values against the
oracle either way."""
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
    yield B
    B.use_torch_allocator()


def _check(bsm, oracle, Ah, Bh, eps, refuse=None):
    """One multiply against the oracle; the sizes it asked the allocator for (`refuse`: answered with no memory)."""
    import torch
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)
    asked = []

    def alloc(n, s):
        asked.append(int(n))
        if int(n) == refuse:
            return None
        return torch.cuda.caching_allocator_alloc(int(n), torch.cuda.current_device(), int(s or 0))

    bsm.set_allocator(alloc, lambda p, n, s: torch.cuda.caching_allocator_delete(p))
    try:
        C = bsm.multiply(1.0, A, B, eps=eps, build_stacks=False)
    finally:
        bsm.use_torch_allocator()
    ref = oracle.multiply(1.0, Ah, Bh, eps=eps)
    rp, ci, bo = C.pattern()
    np.testing.assert_array_equal(rp, ref.C.row_ptr)
    np.testing.assert_array_equal(ci, ref.C.col_idx)
    np.testing.assert_array_equal(bo, ref.C.blk_off)
    p = C.products()
    for x, y in ((p.a, ref.prods.a), (p.b, ref.prods.b), (p.c, ref.prods.c)):
        np.testing.assert_array_equal(x, y)
    assert rel_fro(C.data_host(), ref.C.data) <= 1e-12
    return asked


def _bitmap_bytes(B):
    return 4 * B.nbc * ((B.nbr + 31) // 32)


# around a word and around the 32 words a warp expands at a time; C of 650 x 645 blocks
@pytest.mark.parametrize("nbk", [65, 95, 96, 1023, 1024, 1025])
@pytest.mark.parametrize("eps", [0.0, 1e-9, 1.0])
def test_bitmaps(bsm, oracle, nbk, eps):
    rows, cols = I.uniform_sizes(650, 1), I.uniform_sizes(645, 2)
    inner = I.mixed_sizes(nbk, (1, 2), (0.5, 0.5), seed=3)
    occ = 0.9 if nbk < 100 else 0.12
    Ah, Bh = random_bcsr(rows, inner, occ, seed=91), random_bcsr(inner, cols, occ, seed=92)
    asked = _check(bsm, oracle, Ah, Bh, eps)
    if eps == 1e-9 or (eps == 0.0 and nbk > 1000):   # long enough columns with a threshold, without one
        assert _bitmap_bytes(Bh) in asked


def _columns(nbk, nbc, length, seed):
    """`length` blocks of 1 x 1 in every column."""
    rng = np.random.default_rng(seed)
    rows = np.concatenate([rng.choice(nbk, length, replace=False) for _ in range(nbc)])
    return I.assemble(I.uniform_sizes(nbk, 1), I.uniform_sizes(nbc, 1), rows, np.repeat(np.arange(nbc), length), None,
                      seed=seed)


@pytest.mark.parametrize("eps,length,bitmaps", [(0.0, 93, False), (0.0, 94, True), (1e-9, 41, False), (1e-9, 42, True)])
def test_short_columns_are_walked(bsm, oracle, eps, length, bitmaps):
    """1,200 inner blocks are 38 words a column: 56 blocks more without a threshold, two thirds and 16 with one."""
    Ah, Bh = random_bcsr(I.uniform_sizes(1100, 1), I.uniform_sizes(1200, 1), 0.07, seed=93), _columns(1200, 1000, length, 94)
    assert (_bitmap_bytes(Bh) in _check(bsm, oracle, Ah, Bh, eps)) == bitmaps


@pytest.mark.parametrize("rows,bitmaps", [(81, False), (140, True)])
def test_few_products_are_walked(bsm, oracle, rows, bitmaps):
    """Columns of 66 blocks on average, 4.2e5 and 1.2e6 products."""
    bs, cs, inner = I.uniform_sizes(rows, 1), I.uniform_sizes(rows + 2, 1), I.uniform_sizes(70, 1)
    Ah, Bh = random_bcsr(bs, inner, 0.95, seed=95), random_bcsr(inner, cs, 0.95, seed=96)
    assert (_bitmap_bytes(Bh) in _check(bsm, oracle, Ah, Bh, 1e-9)) == bitmaps


def test_refused_bitmaps_fall_back_to_the_walk(bsm, oracle):
    Ah, Bh = random_bcsr(I.uniform_sizes(1024, 1), I.uniform_sizes(1024, 1), 0.1, seed=97), _columns(1024, 1030, 90, 98)
    for eps in (0.0, 1e-9):
        assert _bitmap_bytes(Bh) in _check(bsm, oracle, Ah, Bh, eps, refuse=_bitmap_bytes(Bh))
