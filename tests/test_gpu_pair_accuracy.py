"""Omega of the FP32 pair sums where a group of 32 sources spans several
filaments: the sums in the group's frame are differences there, and must round no
more than the same sums with the cross products formed per pair. A system of an
ensemble is summed in that second way, so each layout is also run as the first
system of an ensemble, and both are compared with the FP64 form.

The bound: over n = 3S rounding errors of one size the two root mean squares differ
by less than three of their joint standard deviations, a factor 1 + 3 / sqrt(n)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _walks(rng, lengths, vf):
    """Random walks (bond 2.2) centred uniformly in a cube at volume fraction vf."""
    side = (sum(lengths) * 4 / 3 * np.pi / vf) ** (1 / 3)
    out = []
    for n in lengths:
        b = rng.standard_normal((n, 3))
        b *= 2.2 / np.linalg.norm(b, axis=1, keepdims=True)
        w = np.cumsum(b, 0)
        out.append(w - w.mean(0) + rng.uniform(0, side, 3))
    return np.ascontiguousarray(np.concatenate(out))


def _apply(fil, sizes, precision, Y, FT, fil_per_sys=None, schedule=None):
    with fil.Filaments(sizes, fil_per_sys, precision=precision) as m:
        if schedule:
            m.set_pair_schedule(*schedule)
        VW = np.full(FT.shape, np.nan)
        m.mobility_apply(Y, FT, VW)
    return VW


@pytest.mark.parametrize("schedule", [None, (256, 2, 1), (128, 1, 2)])
@pytest.mark.parametrize("lengths", [[1] * 8000, [4] * 2000, [12] * 667, [33] * 242,
                                     [16, 48, 29, 35] * 62, [32] * 250])
def test_omega_rounds_no_more_than_per_pair(lengths, schedule):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(len(lengths))
    S = sum(lengths)
    Y, FT = _walks(rng, lengths, 0.02), rng.standard_normal((S, 6))
    ref = _apply(fil, lengths, fil.FIL_FP64, Y, FT)
    one = _apply(fil, lengths, fil.FIL_PAIR32, Y, FT, schedule=schedule)
    far = np.concatenate([Y, Y[:1]]), np.concatenate([FT, FT[:1]])
    ens = _apply(fil, lengths + [1], fil.FIL_PAIR32, *far, fil_per_sys=[len(lengths), 1])[:S]
    e_one, e_ens = np.linalg.norm((one - ref)[:, 3:]), np.linalg.norm((ens - ref)[:, 3:])
    assert e_one <= (1 + 3 / np.sqrt(3 * S)) * e_ens
