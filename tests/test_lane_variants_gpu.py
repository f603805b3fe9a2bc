"""The warp- and lane-per-block kernels of tiny blocks that the FP64 tensor-core
and Ozaki paths keep on the CUDA cores (GPU): every eligible shape under both
variants, forward with an old C and adjoints, against the oracle."""
import numpy as np
import pytest

from paper_1708_03604_gb300 import inputs as I
from tests.helpers import random_bcsr, rel_fro

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 4, 5, 6)


@pytest.fixture(scope="module")
def bsm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_03604_gb300 import bsm as B
    B.lib()
    return B


@pytest.mark.parametrize("sizes", [SIZES, SIZES + (9,)], ids=["tiny", "with_9"])   # all blocks, or some, by lanes
@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("prec", ["fp64_dmma", "ozaki"])
def test_tiny_blocks(bsm, oracle, prec, variant, sizes):
    import torch
    bs = I.mixed_sizes(120, sizes, [1.0 / len(sizes)] * len(sizes), seed=5)
    Ah, Bh = random_bcsr(bs, bs, 0.1, seed=151), random_bcsr(bs, bs, 0.1, seed=152)
    C0 = random_bcsr(bs, bs, 0.05, seed=153)
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)
    try:
        for m in SIZES:
            for n in SIZES:
                bsm.bsm_set_variant(prec, m, n, variant)
        C = bsm.multiply(1.5, A, B, 0.5, bsm.Matrix.from_host(C0), 1e-3, prec=prec)
        ref = oracle.multiply(1.5, Ah, Bh, eps=1e-3, beta=0.5, Cold=C0).C
        np.testing.assert_array_equal(C.pattern()[1], ref.col_idx)
        assert rel_fro(C.data_host(), ref.data) <= 1e-12
        C = bsm.multiply(1.0, A, B, prec=prec)
        ref = oracle.multiply(1.0, Ah, Bh)
        G = np.random.default_rng(4).standard_normal(ref.C.data_len)
        dA, dB = (torch.empty(len(X.data), dtype=torch.float64, device="cuda") for X in (Ah, Bh))
        bsm.multiply_backward(1.0, C, torch.tensor(G, device="cuda"), A, B, dA, dB, prec=prec)
        for got, want in zip((dA, dB), oracle.multiply_backward(1.0, Ah, Bh, ref.C, G, ref.prods)):
            assert rel_fro(got.cpu().numpy(), want) <= 1e-12
    finally:
        for m in SIZES:
            for n in SIZES:
                bsm.bsm_set_variant(prec, m, n, -1)
