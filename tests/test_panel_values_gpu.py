"""Values at the ends of FP32's range through the tcgen05 row-panel engine
(GPU): the drain converts its compensated pairs to FP64 with integers where it
can and with an FP64 addition elsewhere (zero sums, small compensations).
Block sizes on both sides of a chunk of 8 terms of k."""
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


@pytest.mark.parametrize("s", [1, 7, 8, 9, 16, 17, 23, 24])
def test_single_products_over_the_range(bsm, s):
    """C = alpha A I: every element is hi + lo of one element of A.  The TF32 pieces leave out at most 2^-23 of
    it (11 bits twice, rounded to nearest), the one FP32 addition that is not exact at most 2^-23, alpha 2^-53."""
    bs = I.uniform_sizes(11, s)
    Ah = random_bcsr(bs, bs, 0.5, seed=41)
    rng = np.random.default_rng(42)
    Ah.data = Ah.data * 2.0 ** rng.integers(-90, 120, len(Ah.data))
    Ah.data[::5] = 0.0
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(I.identity(bs))
    for alpha in (1.0, -0.375):
        Cp = bsm.multiply(alpha, A, B, prec="tf32x3_panel")
        assert Cp.engine() == "panel_tcgen05"
        want = alpha * Ah.data
        assert (np.abs(Cp.data_host() - want) <= 2.0 ** -21.9 * np.abs(want)).all()


@pytest.mark.parametrize("s", [5, 8, 9, 16, 17, 24])
@pytest.mark.parametrize("group", [1, 3, 8])
def test_sums_with_and_without_old_blocks(bsm, oracle, s, group):
    """Groups that end inside and at a tile's last k-step, old blocks merged; 1e-6 as for the engine elsewhere."""
    bs = I.uniform_sizes(23, s)
    Ah, Bh, C0 = (random_bcsr(bs, bs, occ, seed=n) for occ, n in ((0.6, 51), (0.6, 52), (0.3, 53)))
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)
    try:
        bsm.bsm_set_tuning("tf32x3_panel", "panel_steps", group)
        Cp = bsm.multiply(1.0, A, B, 0.5, bsm.Matrix.from_host(C0), prec="tf32x3_panel")
    finally:
        bsm.bsm_set_tuning("tf32x3_panel", "panel_steps", -1)
    assert Cp.engine() == "panel_tcgen05"
    assert rel_fro(Cp.data_host(), oracle.multiply(1.0, Ah, Bh, beta=0.5, Cold=C0).C.data) <= 1e-6
