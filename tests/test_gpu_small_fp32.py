"""Small systems in the FP32 modes: up to 160 segments a warp per target in
FP64, the FP32 kernel beyond and where the result overwrites the loads; the
allocation-free apply takes the same way.

Tolerance: up to 160 segments that of an FP64 sum of S terms of magnitude sum B
in any order, (S + 32) 2^-53 B; else C_MIXED FP32 roundings of B
(test_gpu_mobility.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rpy  # noqa: E402

pytestmark = pytest.mark.gpu

C_MIXED = 4 * 32 + 16


@pytest.mark.parametrize("over_loads", [False, True])
@pytest.mark.parametrize("S", [1, 33, 159, 160, 161])
@pytest.mark.parametrize("mode", ["FIL_PAIR32", "FIL_MIXED"])
def test_around_the_largest_size(S, mode, over_loads):
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(S)
    step = rng.standard_normal((S, 3))
    Y = np.cumsum(2.2 * step / np.linalg.norm(step, axis=1, keepdims=True), axis=0)
    FT = rng.standard_normal((S, 6))
    ref, B = rpy.apply(Y, FT, with_abs=True, nthreads=8)
    Yd, Fd = torch.tensor(Y, device="cuda"), torch.tensor(FT, device="cuda")
    out = Fd.clone() if over_loads else torch.full_like(Fd, float("nan"))
    with fil.Filaments([S], precision=getattr(fil, mode)) as m:
        m.mobility_apply(Yd, out if over_loads else Fd, out)
    free = Fd.clone() if over_loads else torch.full_like(Fd, float("nan"))
    fil.fil_rpy_apply_noalloc(S, Yd, free if over_loads else Fd, free)
    torch.cuda.synchronize()
    assert torch.equal(out, free)
    u = (S + 32) * 2.0 ** -53 if S <= 160 and not over_loads else C_MIXED * 2.0 ** -24
    assert np.all(np.abs(out.cpu().numpy() - ref) <= u * B)
