"""What the tuner searches, on the host: the timed multiply is replaced by a
stub on which every trial is faster than the last (what noise can look like), so
whatever is searched is also chosen."""
import numpy as np
import pytest


@pytest.fixture()
def tuner(monkeypatch):
    from types import SimpleNamespace

    from paper_1708_03604_gb300 import autotune, bsm, build
    build.build()
    bsm.lib()
    times = iter(0.9 ** i for i in range(10000))
    monkeypatch.setattr(autotune, "_numeric_ms", lambda *a, **k: next(times))
    monkeypatch.setattr(bsm.Matrix, "empty", lambda *a, **k: None)
    monkeypatch.setattr(bsm, "bsm_set_profiling", lambda on: None)
    sizes = (2, 5, 6)

    def tune(prec, dtype):
        X = SimpleNamespace(row_bs=np.array(sizes), col_bs=np.array(sizes), info=lambda: SimpleNamespace(dtype=dtype))
        try:
            return autotune.tune(X, X, prec=prec, reps=1)
        finally:
            autotune.reset(prec, sizes)
    return tune


DEFAULTS = {"2x2": 1, "2x5": 1, "5x2": 1, "2x6": 1, "6x2": 1, "5x5": 0, "6x6": 0}


def test_variants_are_searched_where_they_choose_a_kernel(tuner):
    from paper_1708_03604_gb300 import bsm
    for prec in ("fp64_dmma", "ozaki"):
        assert tuner(prec, bsm.BSM_FP64)["variants"] == dict.fromkeys(DEFAULTS, 1)
    t = tuner("fp64", bsm.BSM_FP64)
    assert t["variants"] == DEFAULTS and set(t["params"]) == {"fp64_build", "ctas_per_sm", "sched_tile"}
    for prec in ("fp64", "fp64_dmma"):
        t = tuner(prec, bsm.BSM_FP32)
        assert t["variants"] == DEFAULTS and set(t["params"]) == {"ctas_per_sm", "sched_tile"}
