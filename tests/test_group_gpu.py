"""The CUDA-core kernels' lane groups (GPU): output blocks of every layout the
kernel chooses from (a warp per block, several blocks per warp in row- or
column-keeping groups, several passes over large blocks), with enough blocks
that small ones share a warp.  Every element is one chain of FP64 fused
multiply-adds in ascending k whatever the layout, so the builds (which choose
different layouts) must agree bit for bit; against the oracle 1e-12.  FP32
data runs register tiles in lane groups, checked against FP64 data."""
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


def _with_builds(bsm, call):
    """call() under every build the kernel may be asked for; the results must be the same bits."""
    from paper_1708_03604_gb300 import autotune
    got = []
    try:
        for build in (-1, 1, 2):
            bsm.bsm_set_tuning("fp64", "fp64_build", build)
            got.append(call())
    finally:
        autotune.reset("fp64")
    for g in got[1:]:
        for x, y in zip(got[0], g):
            np.testing.assert_array_equal(x, y)
    return got[0]


SHAPES = [(1,), (2,), (3,), (4,), (5,), (6,), (8,), (9,), (13,), (17,), (28,), (4, 1), (5, 13, 23), (3, 7, 16, 32)]


@pytest.mark.parametrize("sizes", SHAPES, ids=lambda s: "_".join(map(str, s)))
def test_layouts_agree_and_match_oracle(bsm, oracle, sizes):
    import torch
    nb = 170 if max(sizes) < 28 else 100
    bs = I.mixed_sizes(nb, sizes, [1.0 / len(sizes)] * len(sizes), seed=5)
    # a few rows of A hold nothing: C blocks there come from the old C alone
    Ah, Bh = random_bcsr(bs, bs, 0.12, seed=21), random_bcsr(bs, bs, 0.12, seed=22)
    C0 = random_bcsr(bs, bs, 0.2, seed=23)
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)

    def plain():
        C = bsm.multiply(1.0, A, B)
        g = torch.linspace(-1.0, 1.0, C.info().data_len, dtype=torch.float64, device="cuda")
        dA = torch.full((len(Ah.data),), np.nan, dtype=torch.float64, device="cuda")
        dB = torch.full((len(Bh.data),), np.nan, dtype=torch.float64, device="cuda")
        bsm.multiply_backward(0.5, C, g, A, B, dA, dB)
        return C.data_host(), dA.cpu().numpy(), dB.cpu().numpy()

    c, dA, dB = _with_builds(bsm, plain)
    ref = oracle.multiply(1.0, Ah, Bh)
    assert rel_fro(c, ref.C.data) <= 1e-12
    G = np.linspace(-1.0, 1.0, ref.C.data_len)
    dA_ref, dB_ref = oracle.multiply_backward(0.5, Ah, Bh, ref.C, G, ref.prods)
    assert rel_fro(dA, dA_ref) <= 1e-12 and rel_fro(dB, dB_ref) <= 1e-12

    def merged():
        return (bsm.multiply(-0.75, A, B, 0.5, bsm.Matrix.from_host(C0), 0.9).data_host(),)

    c, = _with_builds(bsm, merged)
    ref = oracle.multiply(-0.75, Ah, Bh, eps=0.9, beta=0.5, Cold=C0)
    assert rel_fro(c, ref.C.data) <= 1e-12


FP32_SHAPES = [(1,), (3,), (4,), (5,), (8,), (13,), (17,), (24,), (25,), (33,), (4, 1), (5, 13, 23), (3, 7, 16, 32)]


@pytest.mark.parametrize("sizes", FP32_SHAPES, ids=lambda s: "_".join(map(str, s)))
def test_fp32_tiles_within_their_bound(bsm, sizes):
    """FP32 data: one FP32 chain of fused multiply-adds per product and element, the products added in FP64 in
    order.  Every element within the bound of that: k roundings of 2^-24 of the magnitude in the longest product
    and one of the result (doubled: 2^-23), against FP64 data of the same values; the adjoints within 1e-5."""
    import torch
    nb = 150 if max(sizes) < 24 else 100
    bs = I.mixed_sizes(nb, sizes, [1.0 / len(sizes)] * len(sizes), seed=5)
    Ah, Bh = random_bcsr(bs, bs, 0.12, seed=61, dtype=np.float32), random_bcsr(bs, bs, 0.12, seed=62, dtype=np.float32)
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)
    A64, B64 = bsm.Matrix.from_host(Ah.astype(np.float64)), bsm.Matrix.from_host(Bh.astype(np.float64))
    C, C64 = bsm.multiply(1.0, A, B), bsm.multiply(1.0, A64, B64)
    c, c64 = C.data_host().astype(np.float64), C64.data_host()
    # magnitude of every element's terms, from the absolute values
    absA, absB = (bsm.Matrix.from_host(I.BCSR(*(list(vars(X).values())[:5]), np.abs(X.data).astype(np.float64)))
                  for X in (Ah, Bh))
    mag = bsm.multiply(1.0, absA, absB).data_host()
    assert (np.abs(c - c64) <= (max(sizes) + 2) * 2.0 ** -23 * mag).all()
    g64 = torch.linspace(-1.0, 1.0, C.info().data_len, dtype=torch.float64, device="cuda")
    g = g64.float()
    got, ref = [], []
    for out, Cx, Ax, Bx, gx in ((got, C, A, B, g), (ref, C64, A64, B64, g.double())):
        dA, dB = (torch.full((len(X.data),), np.nan, dtype=gx.dtype, device="cuda") for X in (Ah, Bh))
        bsm.multiply_backward(-0.5, Cx, gx, Ax, Bx, dA, dB)
        out += [dA.double().cpu().numpy(), dB.double().cpu().numpy()]
    for x, y in zip(got, ref):
        assert rel_fro(x, y) <= 1e-5


def test_fp32_old_blocks_zero_and_non_finite(bsm):
    """Old blocks merged with beta, zero partial sums (converted the usual way) and infinities, against FP64 data."""
    bs = I.mixed_sizes(120, (5, 8, 23), (0.4, 0.3, 0.3), seed=9)
    Ah, Bh = random_bcsr(bs, bs, 0.1, seed=71), random_bcsr(bs, bs, 0.1, seed=72)
    C0 = random_bcsr(bs, bs, 0.2, seed=73)
    Ah.data[: len(Ah.data) // 3] = 0.0
    Bh.data[-1] = np.inf
    f = np.float32
    Ah.data, Bh.data, C0.data = (X.data.astype(f).astype(np.float64) for X in (Ah, Bh, C0))
    want = bsm.multiply(0.5, *(bsm.Matrix.from_host(X) for X in (Ah, Bh)), 2.0, bsm.Matrix.from_host(C0)).data_host()
    got = bsm.multiply(0.5, *(bsm.Matrix.from_host(X.astype(f)) for X in (Ah, Bh)), 2.0,
                       bsm.Matrix.from_host(C0.astype(f))).data_host().astype(np.float64)
    fin = np.isfinite(want)
    np.testing.assert_array_equal(np.isfinite(got), fin)
    assert rel_fro(got[fin], want[fin]) <= 1e-5


def test_non_finite_values_stay_in_their_rows(bsm):
    """Infinities and NaN reach exactly the elements whose chain holds them (idle lane slots read no other block)."""
    bs = I.uniform_sizes(150, 5)
    Ah, Bh = random_bcsr(bs, bs, 0.1, seed=31), random_bcsr(bs, bs, 0.1, seed=32)
    base = bsm.multiply(1.0, bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)).to_host()
    Ah.data[7], Ah.data[1003] = np.inf, np.nan
    got = bsm.multiply(1.0, bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)).to_host()
    brow = np.repeat(np.arange(150), np.diff(Ah.row_ptr))
    bad = {(int(brow[e // 25]), (e % 25) // 5) for e in (7, 1003)}
    crow = np.repeat(np.arange(150), np.diff(got.row_ptr))
    rows = np.stack([np.repeat(crow, 25), np.tile(np.arange(25) // 5, len(crow))], 1)
    hit = np.array([(int(i), int(r)) in bad for i, r in rows])
    np.testing.assert_array_equal(got.data[~hit], base.data[~hit])
    assert not np.isfinite(got.data[hit]).all()


@pytest.mark.parametrize("prec", ["fp64", "fp64_dmma"])
def test_fp32_sums_per_variant(bsm, prec):
    """FP32 data with flush_every above 1: variant 1 (the default up to 16 elements, on request for 5 x 5 and 6 x 6
    blocks) adds every product in FP64, bit for bit what flush_every = 1 gives; variant 0 adds them together."""
    import torch
    sizes = (2, 4, 5, 6)
    bs = I.mixed_sizes(120, sizes, [0.25] * 4, seed=5)
    Ah, Bh = random_bcsr(bs, bs, 0.3, seed=63, dtype=np.float32), random_bcsr(bs, bs, 0.3, seed=64, dtype=np.float32)
    A, B = bsm.Matrix.from_host(Ah), bsm.Matrix.from_host(Bh)

    def run(flush):
        C = bsm.multiply(1.0, A, B, prec=prec, flush_every=flush)
        g = torch.linspace(-1.0, 1.0, C.info().data_len, dtype=torch.float32, device="cuda")
        dA, dB = (torch.empty(len(X.data), dtype=torch.float32, device="cuda") for X in (Ah, Bh))
        bsm.multiply_backward(1.0, C, g, A, B, dA, dB, prec=prec, flush_every=flush)
        rc = np.stack([np.repeat(bs, np.diff(C.pattern()[0])), bs[C.pattern()[1]]], 1)
        shape = np.repeat(rc, rc[:, 0] * rc[:, 1], axis=0)
        return C.data_host(), shape, dA.cpu().numpy(), dB.cpu().numpy()

    def among(shape, keys):
        return np.array([tuple(s) in keys for s in shape.tolist()])

    try:
        one, shape, dA1, dB1 = run(1)
        default = run(8)[0]
        tiny = shape[:, 0] * shape[:, 1] <= 16
        square = among(shape, {(5, 5), (6, 6)})
        np.testing.assert_array_equal(default[tiny], one[tiny])
        assert (default[square] != one[square]).any()      # eight products share an FP32 sum
        for m, n in ((5, 5), (6, 6)):
            bsm.bsm_set_variant(prec, m, n, 1)
        got, _, dA, dB = run(8)
        np.testing.assert_array_equal(got[tiny | square], one[tiny | square])
        for x, y, X in ((dA, dA1, Ah), (dB, dB1, Bh)):     # the adjoints' blocks, by their own shapes
            rc = np.stack([np.repeat(bs, np.diff(X.row_ptr)), bs[X.col_idx]], 1)
            s = np.repeat(rc, rc[:, 0] * rc[:, 1], axis=0)
            keep = (s[:, 0] * s[:, 1] <= 16) | among(s, {(5, 5), (6, 6)})
            np.testing.assert_array_equal(x[keep], y[keep])
        bsm.bsm_set_variant(prec, 4, 4, 0)
        got = run(8)[0]
        four = among(shape, {(4, 4)})
        assert (got[four] != one[four]).any()
    finally:
        for m, n in ((4, 4), (5, 5), (6, 6)):
            bsm.bsm_set_variant(prec, m, n, -1)


def test_fp32_reports_no_fp64_build(bsm):
    """The launch configuration names a build for FP64 data only."""
    bs = I.mixed_sizes(60, (5, 13), (0.5, 0.5), seed=9)
    Ah = random_bcsr(bs, bs, 0.2, seed=74)
    for X, build in ((Ah, 1), (Ah.astype(np.float32), -1)):
        A = bsm.Matrix.from_host(X)
        cfg = bsm.multiply(1.0, A, A).launch_config()
        assert cfg["kernel"] == "fp64_cores" and cfg["fp64_build"] == build and cfg["grid"] > 0
