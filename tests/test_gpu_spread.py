"""The order of the groups' records that mid-size FP32 systems use (48 to 384
groups of 32 segments): the smallest and largest such system, one group less and
more, and remainders of the 16 runs, with filaments whose close pairs lie in
neighbouring groups; against the oracle on sampled rows, within the bound of
test_gpu_mobility.py (C_MIXED roundings of the magnitude sum)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rpy  # noqa: E402

pytestmark = pytest.mark.gpu

C_MIXED = 4 * 32 + 16


@pytest.mark.parametrize("S", [1504, 1505, 1537, 2047, 12257, 12288, 12289])
def test_rows(S):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(S)
    step = rng.standard_normal((S, 3))
    Y = np.cumsum(2.2 * step / np.linalg.norm(step, axis=1, keepdims=True), axis=0)
    FT = rng.standard_normal((S, 6))
    rows = np.unique(np.concatenate([[0, 31, 32, 63, 64, S - 2, S - 1],
                                     rng.integers(0, S, size=200)]))
    ref, B = rpy.apply_rows(Y, FT, rows, with_abs=True, nthreads=8)
    segs = [S // 4] * 3 + [S - 3 * (S // 4)]
    with fil.Filaments(segs, precision=fil.FIL_MIXED, max_iter=1) as m:
        VW = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW)
    assert np.all(np.isfinite(VW))
    assert np.all(np.abs(VW[rows] - ref) <= C_MIXED * 2.0 ** -24 * B)
