"""FP64 applies of one system with a segment so far away that r^2 overflows: its
pairs add nothing (the far form tends to zero), so the others' rows are those of
the system without it, and its own are its self mobility, within the summation
bound of test_gpu_pair64.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rpy  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [20, 1100])
def test_overflowing_distance(S):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(S)
    Y, FT = rng.uniform(0, 60, size=(S, 3)), rng.standard_normal((S, 6))
    ref, B = rpy.apply(Y[:-1].copy(), FT[:-1].copy(), with_abs=True)
    Y[-1] = 1e160
    with fil.Filaments([S], precision=fil.FIL_FP64) as m:
        VW = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW)
    tol = (S + 32) * 2.0 ** -53
    assert np.all(np.abs(VW[:-1] - ref) <= tol * B)
    own = FT[-1] / (8 * np.pi) * np.array([4 / 3] * 3 + [1.0] * 3)
    assert np.all(np.abs(VW[-1] - own) <= tol * np.abs(own))
