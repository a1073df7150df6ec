"""The automatic schedule of the FP32 pair kernel (64-target tiles, the units
(tile, 32-source group) split over the warps of one CTA per SM) at its edges:
sizes around a tile, a group and the point where every warp has one unit, and
systems of an ensemble that share a grid, against the oracle and within the
bound of test_gpu_mobility.py (C_MIXED roundings of the magnitude sum)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rpy  # noqa: E402

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24
C_MIXED = 4 * 32 + 16


def _lines(rng, S, spacing=2.2):
    """Straight lines of 32 touching-free segments at random places (the groups
    of 32 sources are then as long as they get), cut at S segments."""
    m = -(-S // 32)
    t = rng.standard_normal((m, 3))
    t /= np.linalg.norm(t, axis=1, keepdims=True)
    base = rng.uniform(0, 12.0 * m ** (1 / 3) + 20, size=(m, 3))
    return np.ascontiguousarray(
        (base[:, None] + spacing * np.arange(32)[None, :, None] * t[:, None]).reshape(-1, 3)[:S])


@pytest.mark.parametrize("S", [1, 31, 33, 64, 65, 96, 127, 1889, 3457])
def test_sizes_around_tiles_and_groups(S):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(S)
    Y, FT = _lines(rng, S), rng.standard_normal((S, 6))
    ref, B = rpy.apply(Y, FT, with_abs=True, nthreads=8)
    with fil.Filaments([S], precision=fil.FIL_PAIR32) as m:
        VW = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW)
        VW2 = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW2)
    np.testing.assert_array_equal(VW, VW2)
    assert np.all(np.abs(VW - ref) <= C_MIXED * U32 * B)


@pytest.mark.parametrize("sizes", [[1, 64, 65, 200], [33] * 40, [700, 1, 1300, 31]])
def test_systems_of_an_ensemble(sizes):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(sum(sizes))
    S = sum(sizes)
    Y = np.concatenate([_lines(rng, n) for n in sizes])
    FT = rng.standard_normal((S, 6))
    with fil.Filaments(sizes, [1] * len(sizes), precision=fil.FIL_MIXED) as m:
        VW = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW)
    at = 0
    for n in sizes:
        ref, B = rpy.apply(Y[at:at + n], FT[at:at + n], with_abs=True)
        assert np.all(np.abs(VW[at:at + n] - ref) <= C_MIXED * U32 * B)
        at += n
