"""The FP64 applies of one system that read the caller's arrays (a warp per
target; every unordered pair once in 64-segment tiles) at the edges of their
ranges and tiles, against the oracle; and a result that overwrites an input.

Tolerance: a component is a sum of S pair terms of magnitude sum B, summed in
FP64 in some order with a few roundings per term: |error| <= (S + 32) 2^-53 B
covers any order."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rpy  # noqa: E402

pytestmark = pytest.mark.gpu


def _inputs(S, seed):
    """Random walks: bonded and overlapping neighbours, distant pairs, and two
    coincident segments."""
    rng = np.random.default_rng(seed)
    step = rng.standard_normal((S, 3))
    Y = np.cumsum(2.2 * step / np.linalg.norm(step, axis=1, keepdims=True), axis=0)
    Y += rng.uniform(0, 40, size=(-(-S // 32), 3)).repeat(32, axis=0)[:S]
    if S > 3:
        Y[S // 2] = Y[S // 3]
    return np.ascontiguousarray(Y), rng.standard_normal((S, 6))


@pytest.mark.parametrize("S", [1, 2, 31, 32, 33, 65, 1023, 1024, 1025, 1088, 1089, 2111])
def test_sizes(S):
    from paper_1903_12609_gb300 import fil
    Y, FT = _inputs(S, S)
    ref, B = rpy.apply(Y, FT, 1.2, 0.7, with_abs=True, nthreads=8)
    with fil.Filaments([S], a=1.2, eta=0.7, precision=fil.FIL_FP64) as m:
        VW = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW)
        again = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, again)
    np.testing.assert_array_equal(VW, again)
    assert np.all(np.abs(VW - ref) <= (S + 32) * 2.0 ** -53 * B)


@pytest.mark.parametrize("S", [8192, 8193])
def test_largest_size_of_the_slots_and_the_next(S):
    from paper_1903_12609_gb300 import fil
    Y, FT = _inputs(S, 7)
    rows = np.array([0, 1, 63, 64, 4095, 8127, 8128, S - 1])
    ref, B = rpy.apply_rows(Y, FT, rows, with_abs=True, nthreads=8)
    with fil.Filaments([4096, S - 4096], precision=fil.FIL_FP64, max_iter=1) as m:
        VW = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW)
    assert np.all(np.abs(VW[rows] - ref) <= (S + 32) * 2.0 ** -53 * B)


@pytest.mark.parametrize("S", [20, 1500])
def test_result_over_the_loads(S):
    """VW may be the array of the loads: the apply reads them all first."""
    from paper_1903_12609_gb300 import fil
    Y, FT = _inputs(S, 3)
    Yd, FTd = torch.from_numpy(Y).cuda(), torch.from_numpy(FT).cuda()
    out = torch.empty_like(FTd)
    with fil.Filaments([S], precision=fil.FIL_FP64) as m:
        m.mobility_apply(Yd, FTd, out)
        m.mobility_apply(Yd, FTd, FTd)
        torch.cuda.synchronize()
    ref, B = rpy.apply(Y, FT, with_abs=True)
    for got in (out.cpu().numpy(), FTd.cpu().numpy()):
        assert np.all(np.abs(got - ref) <= (S + 32) * 2.0 ** -53 * B)
