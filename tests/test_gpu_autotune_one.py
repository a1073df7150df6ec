"""fil_autotune on contexts of one system: it may change the order of the pair terms, not
the precision they are summed in."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rpy  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [20, 100, 160, 161, 700])
@pytest.mark.parametrize("mode", ["FIL_PAIR32", "FIL_MIXED", "FIL_FP64"])
def test_tuning_keeps_the_precision(S, mode):
    """Up to 160 segments, and in FP64, an FP64 sum of S terms in any order,
    (S + 32) 2^-53 of the magnitude sum; else 144 FP32 roundings (test_gpu_mobility.py)."""
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(S)
    step = rng.standard_normal((S, 3))
    Y = np.cumsum(2.2 * step / np.linalg.norm(step, axis=1, keepdims=True), axis=0)
    FT = rng.standard_normal((S, 6))
    ref, B = rpy.apply(Y, FT, with_abs=True, nthreads=8)
    with fil.Filaments([S], precision=getattr(fil, mode)) as m:
        m.set_state(Y, np.tile([1.0, 0.0, 0.0, 0.0], (S, 1)))
        tile, ctas, ms = m.autotune(20)
        assert tile in (128, 256) and ctas >= 1 and ms > 0
        assert m.pair_schedule()[0] == tile and m.pair_schedule()[2] == ctas
        VW = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW)
    u = (S + 32) * 2.0 ** -53 if S <= 160 or mode == "FIL_FP64" else 144 * 2.0 ** -24
    assert np.all(np.abs(VW - ref) <= u * B)
