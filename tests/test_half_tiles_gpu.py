"""The split paths' half tiles (GPU): where at most 8 rows of an output block
fall into its last tile row, the packs, copies and sums of the empty half fall
away.  Heights on both sides of every edge.  Against the oracle the bound of the
path (1e-6, the two-piece BF16 split 1e-4); kernels for blocks of one height
class and the one for any height run every element through the same chain of
sums, so they must agree bit for bit (one block product a sum)."""
import numpy as np
import pytest

from paper_1708_03604_gb300 import inputs as I
from tests.helpers import random_bcsr, rel_fro

pytestmark = pytest.mark.gpu

TOL = {"tf32x3": 1e-6, "bf16x6": 1e-6, "bf16x3": 1e-4}


@pytest.fixture(scope="module")
def bsm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_03604_gb300 import bsm as B
    B.lib()
    return B


@pytest.mark.parametrize("heights", [(5, 8, 9), (16, 17, 24), (23, 25, 32), (33, 40, 41), (48, 56, 7)], ids=str)
@pytest.mark.parametrize("prec", sorted(TOL))
def test_heights(bsm, oracle, prec, heights):
    from paper_1708_03604_gb300 import autotune
    rows = I.mixed_sizes(40, heights, [1 / 3] * 3, seed=3)
    mid = I.mixed_sizes(40, (3, 8, 17), [1 / 3] * 3, seed=4)
    cols = I.mixed_sizes(40, (6, 13, 24), [1 / 3] * 3, seed=5)
    Ah, Bh = random_bcsr(rows, mid, 0.3, seed=6), random_bcsr(mid, cols, 0.3, seed=7)
    C0 = random_bcsr(rows, cols, 0.4, seed=8)
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)
    ref = oracle.multiply(1.5, Ah, Bh, 0.5, C0)
    for flush in (0, 1, -3, 4):
        got = {}
        try:
            for pm in (-1, 2, 1):
                bsm.bsm_set_tuning(prec, "pass_mt", pm)
                got[pm] = bsm.multiply(1.5, A, B, 0.5, bsm.Matrix.from_host(C0), prec=prec, flush_every=flush).data_host()
        finally:
            autotune.reset(prec)
        for pm, c in got.items():
            assert rel_fro(c, ref.C.data) <= TOL[prec], (flush, pm)
            if flush in (0, 1):
                np.testing.assert_array_equal(c, got[-1])


@pytest.mark.parametrize("flush", [0, 1, 4, -3])
@pytest.mark.parametrize("prec", sorted(TOL))
def test_classes(bsm, oracle, prec, flush):
    """Enough blocks (22,500) for an instance per height class.  With more than one block product a sum the one-row
    instances add in two accumulators and the two-row ones in one, so blocks of one tile row must be the bits of the
    any-height instance of one row, the others of that of two; with one product a sum all three agree."""
    from paper_1708_03604_gb300 import autotune
    rows = I.mixed_sizes(150, (5, 8, 9, 16, 17, 24, 25, 40), [1 / 8] * 8, seed=3)
    mid, cols = I.mixed_sizes(60, (3, 8, 17), [1 / 3] * 3, seed=4), I.mixed_sizes(150, (6, 13, 24), [1 / 3] * 3, seed=5)
    Ah, Bh = random_bcsr(rows, mid, 0.4, seed=6), random_bcsr(mid, cols, 0.4, seed=7)
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)
    got = {}
    try:
        for pm in (-1, 2, 1):
            bsm.bsm_set_tuning(prec, "pass_mt", pm)
            C = bsm.multiply(1.0, A, B, prec=prec, flush_every=flush)
            got[pm] = C.data_host()
            if pm == -1:
                assert C.launch_config()["pass_mt"] == 0
    finally:
        autotune.reset(prec)
    rp, ci, _ = C.pattern()
    m, n = np.repeat(rows, np.diff(rp)), cols[ci]
    low = np.repeat(m <= 16, m * n)
    np.testing.assert_array_equal(got[-1][low], got[1][low])
    np.testing.assert_array_equal(got[-1][~low], got[2][~low])
    if flush in (0, 1):
        np.testing.assert_array_equal(got[1], got[2])
        assert rel_fro(got[-1], oracle.multiply(1.0, Ah, Bh).C.data) <= TOL[prec]
