"""One system's FP32 apply under the automatic schedule (two targets packed in a lane)
and under schedules set by hand, whose grids fill the SMs or leave room: sizes around a
lane's two slots and a group's even and odd sources, against the oracle and within
the bound of test_gpu_mobility.py (144 roundings of the magnitude sum)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rpy  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [161, 191, 193, 224, 225, 1505, 1537])
def test_schedules_of_one_system(S):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(S)
    # random walks, every third segment moved away: overlapping, close and far pairs
    step = rng.standard_normal((S, 3))
    Y = np.cumsum(2.2 * step / np.linalg.norm(step, axis=1, keepdims=True), axis=0)
    Y[::3] += rng.uniform(0, 60, size=Y[::3].shape)
    FT = rng.standard_normal((S, 6))
    ref, B = rpy.apply(Y, FT, with_abs=True, nthreads=8)
    with fil.Filaments([S], precision=fil.FIL_PAIR32) as m:
        for schedule in (None, (256, 2, 1), (256, 2, 4), (128, 1, 6)):
            if schedule:
                m.set_pair_schedule(*schedule)
            VW = np.full((S, 6), np.nan)
            m.mobility_apply(Y, FT, VW)
            assert np.all(np.abs(VW - ref) <= 144 * 2.0 ** -24 * B), schedule
