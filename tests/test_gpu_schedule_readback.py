"""A pair schedule that was read from a context of one system and is set again is the one
that ran: the apply keeps its bits, also after another schedule in between."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [30, 160, 161, 1000, 1500])
@pytest.mark.parametrize("mode", ["FIL_PAIR32", "FIL_FP64"])
def test_reported_schedule_set_again(S, mode):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(S)
    Y, FT = rng.uniform(0, 3.0 * S ** (1 / 3), (S, 3)), rng.standard_normal((S, 6))

    def apply(m):
        VW = np.full((S, 6), np.nan)
        m.mobility_apply(Y, FT, VW)
        return VW

    with fil.Filaments([S], precision=getattr(fil, mode)) as m:
        first, schedule = apply(m), m.pair_schedule()
        m.set_source_split(m.source_split())
        np.testing.assert_array_equal(apply(m), first)
        m.set_pair_schedule(*schedule)
        assert m.pair_schedule() == schedule and m.source_split() == 1
        np.testing.assert_array_equal(apply(m), first)
        m.set_pair_schedule(128, 1, 1)
        apply(m)
        m.set_pair_schedule(*schedule)
        np.testing.assert_array_equal(apply(m), first)
