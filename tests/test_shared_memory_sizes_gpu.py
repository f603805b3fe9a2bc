"""Launches whose dynamic shared memory ends just below 48 KB (GPU): a kernel's
static and dynamic arrays share that limit unless it opts in to more, so each of
these sizes needs the opt-in although its dynamic part alone does not.  Sizes
step through the last 2 KB below the limit for every kernel that sizes its
arrays from the operands; results exactly those of 1 x 1 blocks (products of two
small integers) or the oracle's."""
import ctypes

import numpy as np
import pytest

from paper_1708_03604_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bsm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_03604_gb300 import bsm as B
    B.lib()
    return B


def _ones(nbr, nbc, rows, cols):
    """1 x 1 blocks of small integers."""
    X = I.assemble(I.uniform_sizes(nbr, 1), I.uniform_sizes(nbc, 1), rows, cols, None, seed=1)
    X.data[:] = np.arange(len(X.data)) % 7 + 1.0
    return X


# words of shared memory: 2 ceil(N / 32) + N and the inner dimension's part, one word or the bitmaps' lists
@pytest.mark.parametrize("lo,hi", [(7140, 7270), (11430, 11600)])
def test_fill_by_columns(bsm, lo, hi):
    A = bsm.Matrix.from_host(_ones(1, 1, [0], [0]))
    for n in range(lo, hi, 12):
        Bh = _ones(1, n, np.zeros(n, np.int64), np.arange(n))
        C = bsm.multiply(1.0, A, bsm.Matrix.from_host(Bh))
        np.testing.assert_array_equal(C.data_host(), Bh.data)


def test_fill_by_rows(bsm):
    nbk = 60000        # A's map over the inner dimension does not fit: no columns
    Ah = _ones(1, nbk, np.zeros(2, np.int64), [0, nbk - 1])
    A = bsm.Matrix.from_host(Ah)
    for n in range(1340, 1360):   # 2 ceil(n / 32) + 9 n + 1 words: 12,288 are 48 KB
        Bh = _ones(nbk, n, np.full(n, nbk - 1), np.arange(n))
        C = bsm.multiply(1.0, A, bsm.Matrix.from_host(Bh))
        np.testing.assert_array_equal(C.data_host(), Ah.data[1] * Bh.data)


def test_counts(bsm):
    import torch
    A = bsm.Matrix.from_host(_ones(1, 1, [0], [0]))
    for words in (11900, 12000, 12100, 12200, 12288):   # a bit per block column of C
        n = 32 * words
        Bh = _ones(1, n, [0, 0, 0], [0, n // 2, n - 1])
        B = bsm.Matrix.from_host(Bh)
        C = bsm.multiply(1.0, A, B)
        np.testing.assert_array_equal(C.pattern()[1], Bh.col_idx)
        np.testing.assert_array_equal(C.data_host(), Bh.data)
        out = torch.zeros(5, dtype=torch.int64, device="cuda")
        p = out.data_ptr()
        bsm._sync_stream()
        assert bsm.lib().bsm_count_products_static(A.h, B.h, 0.0, ctypes.c_void_p(p), ctypes.c_void_p(p + 8),
                                                   ctypes.c_void_p(p + 16)) == bsm.BSM_OK
        torch.cuda.synchronize()
        assert out.tolist() == [3, 3, 3, 0, 3]


@pytest.mark.parametrize("nb", [17440, 17600, 17856])
def test_panel_steps(bsm, oracle, nb):
    """The row-panel engine's k-step bitmaps: 88 bytes for every 32 inner blocks."""
    d = np.arange(nb)
    off = np.concatenate([d, d[1:], d[:-1]])
    cols = np.concatenate([d, d[:-1], d[1:]])
    bs = I.uniform_sizes(nb, 2)
    Ah, Bh = (I.assemble(bs, bs, off, cols, None, seed=s) for s in (5, 6))
    C = bsm.multiply(1.0, bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh), prec="tf32x3_panel")
    assert C.engine() == "panel_tcgen05"
    ref = oracle.multiply(1.0, Ah, Bh).C
    np.testing.assert_array_equal(C.pattern()[1], ref.col_idx)
    assert np.linalg.norm(C.data_host() - ref.data) <= 1e-6 * np.linalg.norm(ref.data)
