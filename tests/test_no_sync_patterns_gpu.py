"""No-sync calls whose recomputed pattern has the eager call's sizes but other
blocks in the same places (GPU): new values move the filter's decisions from one
block to another.  The order, groups and variant marks of the numeric kernels
come from the eager call, the column copy of B from an earlier pattern of it; the
result must be the new pattern's, against the oracle."""
import numpy as np
import pytest

from paper_1708_03604_gb300 import inputs as I
from tests.helpers import random_bcsr, rel_fro

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp64_dmma": 1e-12, "tf32x3": 1e-6, "bf16x6": 1e-6, "bf16x3": 1e-4, "ozaki": 1e-13}


@pytest.fixture(scope="module")
def bsm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_03604_gb300 import bsm as B
    B.lib()
    return B


def _block_values(X, seed, on):
    """X with blocks of norm about 1 where `on`, far below the threshold elsewhere."""
    Y = I.BCSR(X.row_bs, X.col_bs, X.row_ptr, X.col_idx, X.blk_off, X.data.copy())
    size = np.diff(np.append(X.blk_off, len(X.data)))
    scale = np.repeat(np.where(on, 1.0 / np.sqrt(size), 1e-8), size)
    rng = np.random.default_rng(seed)
    Y.data[:] = rng.uniform(0.5, 1.5, len(X.data)) * rng.choice([-1.0, 1.0], len(X.data)) * scale
    return Y


def _full(rows, cols):
    r, c = np.divmod(np.arange(len(rows) * len(cols)), len(cols))
    return I.assemble(rows, cols, r, c, None, seed=1)


# heights of the block rows: every height class twice, and tiny blocks (3 columns) beside large ones
@pytest.mark.parametrize("heights", [(5, 23, 40, 13), (8, 9), (17, 16, 32), (2, 23), (1, 4, 40)], ids=str)
@pytest.mark.parametrize("prec", sorted(TOL))
def test_blocks_of_other_shapes(bsm, oracle, prec, heights):
    rows = np.array(heights * 2, np.int32)                 # rows i and i + n have one height
    n = len(heights)
    inner, cols = np.array([7, 16], np.int32), np.array([3, 6, 24], np.int32)
    Ah, Bh = _full(rows, inner), random_bcsr(inner, cols, 1.0, seed=2)
    # kept in the eager call: row q of the first or of the second n; then the other one
    first = np.arange(n) % 2 == 0
    keep = np.concatenate([first, ~first])
    on = [np.repeat(k, len(inner)) for k in (keep, ~keep)]
    A1, A2 = (_block_values(Ah, s, o) for s, o in zip((3, 4), on))
    A, B = bsm.Matrix.from_host(A1), bsm.Matrix.from_host(Bh)
    for flush in (0, 4):
        C = bsm.multiply(1.5, A, B, eps=1e-3, prec=prec, flush_every=flush)
        for X in (A2, A1):
            A.set_data(X.data)
            bsm.multiply(1.5, A, B, Cm=C, eps=1e-3, prec=prec, flush_every=flush, no_sync=True)
            ref = oracle.multiply(1.5, X, Bh, eps=1e-3).C
            assert bsm.bsm_get_status(C.h) == 0
            rp, ci, _ = C.pattern()
            np.testing.assert_array_equal(rp, ref.row_ptr)
            np.testing.assert_array_equal(ci, ref.col_idx)
            # (flush_every 4 of the two-piece paths: four products share an FP32 sum)
            assert rel_fro(C.data_host(), ref.data) <= (TOL[prec] if flush == 0 else 2 * TOL[prec])


# B = X + 0 by a filtered add: X holds two patterns, the second one block column further, and the values choose
@pytest.mark.parametrize("rows,inner,cols,occ", [(9, 40, 37, 0.1), (300, 200, 300, 0.3)], ids=["walk", "bitmaps_with_eps"])
@pytest.mark.parametrize("eps", [0.0, 1e-9])
def test_pattern_of_b(bsm, oracle, rows, inner, cols, occ, eps):
    one = random_bcsr(I.uniform_sizes(inner, 2), I.uniform_sizes(cols, 1), occ, seed=11)
    mask = np.zeros((inner, cols), bool)
    mask[np.repeat(np.arange(inner), np.diff(one.row_ptr)), one.col_idx] = True
    mask[0] = True                              # every column has a block in both
    moved = np.roll(mask, 1, axis=1)
    r, c = np.nonzero(mask | moved)
    both = I.assemble(one.row_bs, one.col_bs, r, c, None, seed=12)
    X1, X2 = (_block_values(both, s, m[r, c]) for s, m in ((13, mask), (14, moved)))
    Y = I.BCSR(both.row_bs, both.col_bs, both.row_ptr, both.col_idx, both.blk_off, np.zeros_like(both.data))
    Ah = random_bcsr(I.uniform_sizes(rows, 3), one.row_bs, 1.0, seed=15)

    def kept(X, m):
        z = I.assemble(X.row_bs, X.col_bs, *np.nonzero(m), None, seed=1)
        z.data[:] = X.data.reshape(-1, 2)[m[r, c]].reshape(-1)
        return oracle.multiply(1.0, Ah, z, eps=eps).C

    refs = kept(X1, mask), kept(X2, moved)
    A, X, Ym = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(X1), bsm.Matrix.from_host(Y)
    Z = bsm.add(1.0, X, 1.0, Ym, eps=1e-3)
    C = bsm.multiply(1.0, A, Z, eps=eps)
    assert (C.counts().products >= 1 << 19) == (rows == 300)
    for v, ref in ((X1, refs[0]), (X2, refs[1]), (X1, refs[0]), (X2, refs[1])):
        X.set_data(v.data)
        bsm.add(1.0, X, 1.0, Ym, Z=Z, eps=1e-3, no_sync=True)
        bsm.multiply(1.0, A, Z, Cm=C, eps=eps, no_sync=True)
        assert bsm.bsm_get_status(Z.h) == 0 and bsm.bsm_get_status(C.h) == 0
        for D in (C, bsm.multiply(1.0, A, Z, eps=eps)):          # and an eager call on the rewritten B
            rp, ci, _ = D.pattern()
            np.testing.assert_array_equal(rp, ref.row_ptr)
            np.testing.assert_array_equal(ci, ref.col_idx)
            assert rel_fro(D.data_host(), ref.data) <= 1e-12
