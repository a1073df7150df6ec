"""The ensembles' FP32 pair kernel where a warp's second slot of targets is empty
(the last 256-target tile of a system holds at most 128 + 32 w), where whole warps
are, and where a group has padding sources, in each of its schedules, against the
oracle and within the bound of test_gpu_mobility.py (144 roundings of the magnitude
sum)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rpy  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [1, 31, 97, 128, 129, 160, 161, 255, 256, 257, 289, 384, 385, 640]


@pytest.mark.parametrize("schedule", [None, (256, 2, 1), (128, 1, 3), "split"])
def test_systems_around_the_slots(schedule):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(11)
    S = sum(SIZES)
    # random walks: bonded and overlapping neighbours in every group
    step = rng.standard_normal((S, 3))
    Y = np.cumsum(2.2 * step / np.linalg.norm(step, axis=1, keepdims=True), axis=0)
    FT = rng.standard_normal((S, 6))
    with fil.Filaments(SIZES, [1] * len(SIZES), precision=fil.FIL_MIXED) as m:
        if schedule == "split":
            m.set_pair_schedule(128, 1, 2)
            m.set_source_split(2)
        elif schedule:
            m.set_pair_schedule(*schedule)
        VW = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW)
        again = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, again)
    np.testing.assert_array_equal(VW, again)
    at = 0
    for n in SIZES:
        ref, B = rpy.apply(Y[at:at + n].copy(), FT[at:at + n].copy(), with_abs=True)
        assert np.all(np.abs(VW[at:at + n] - ref) <= 144 * 2.0 ** -24 * B)
        at += n
