"""The FP32 pair kernel of the automatic schedule (64-target tiles per warp, units of 32
sources, 12 warps per SM) at its edges. Up to 160 segments it runs only where the result
overwrites the loads, so the small sizes are reached that way; beyond, sizes around
multiples of a group and a tile, and around the point where every warp of the grid has
one unit. Bound of test_gpu_mobility.py: 144 roundings of the magnitude sum."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rpy  # noqa: E402

pytestmark = pytest.mark.gpu


def _check(S, over_loads):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(S)
    # filaments of 40 in random walks: groups of one filament and of two
    m = -(-S // 40)
    b = rng.standard_normal((m, 40, 3))
    b *= 2.2 / np.linalg.norm(b, axis=2, keepdims=True)
    Y = (np.cumsum(b, 1) + rng.uniform(0, 20.0 * m ** (1 / 3), (m, 1, 3))).reshape(-1, 3)[:S]
    FT = rng.standard_normal((S, 6))
    ref, B = rpy.apply(Y, FT, with_abs=True, nthreads=8)
    Yd, Fd = torch.tensor(Y, device="cuda"), torch.tensor(FT, device="cuda")
    out = Fd if over_loads else torch.full_like(Fd, float("nan"))
    with fil.Filaments([1] * S, precision=fil.FIL_PAIR32) as c:
        c.mobility_apply(Yd, Fd, out)
    torch.cuda.synchronize()
    assert np.all(np.abs(out.cpu().numpy() - ref) <= 144 * 2.0 ** -24 * B)


@pytest.mark.parametrize("S", [1, 2, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129])
def test_small_systems(S):
    _check(S, True)


@pytest.mark.parametrize("S", [161, 192, 223, 255, 256, 257, 319, 321])
def test_tiles_and_groups(S):
    _check(S, False)


@pytest.mark.parametrize("over", [-1, 0, 1])
def test_one_unit_per_warp(over):
    """The largest size whose (tile, group) units are at most the warps of the grid."""
    warps = 12 * torch.cuda.get_device_properties(0).multi_processor_count
    S = 64
    while -(-(S + 1) // 64) * -(-(S + 1) // 32) <= warps:
        S += 1
    _check(S + over, False)
