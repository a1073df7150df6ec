"""The warm-start network's loss where its squares leave FP32's range: a network of
zero weights predicts zeros, so the loss of targets t is sum t^2 / (2 B) exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as om  # noqa: E402

pytestmark = pytest.mark.gpu

NIN = om.DIMS[0][0]


def _loss(t):
    from paper_1903_12609_gb300 import fil
    B = t.shape[0]
    m = fil.fil_mlp_create(B)
    fil.fil_mlp_set_params(m, np.zeros(om.NPARAM, np.float32))
    fil.fil_mlp_set_norm(m, *(np.full(n, v, np.float32) for n, v in
                              ((NIN, 0.0), (NIN, 1.0), (192, 0.0), (192, 1.0))))
    x = torch.zeros(B, NIN, device="cuda")
    loss = fil.fil_mlp_gradients(m, x, torch.from_numpy(t).cuda(), B,
                                 torch.empty(om.NPARAM, device="cuda"))
    fil.fil_mlp_destroy(m)
    return loss


@pytest.mark.parametrize("B", [1, 33, 1024])
@pytest.mark.parametrize("scale", [1e-21, 1e-15, 1e-12, 1.0, 1e18])
def test_every_scale(B, scale):
    """Within the rounding of the FP32 result (FP64 sums of exact squares), half a unit
    of the smallest FP32 number included."""
    t = (scale * np.random.default_rng(B).uniform(0.5, 2.0, (B, 192))).astype(np.float32)
    ref = (t.astype(np.float64) ** 2).sum() / (2 * B)
    assert abs(_loss(t) - ref) <= 2.0 ** -23 * ref + 2.0 ** -149


def test_one_large_residual():
    """One square above FP32's largest number, the loss below it."""
    t = np.ones((1024, 192), np.float32)
    t[700, 5] = 1e20
    ref = (t.astype(np.float64) ** 2).sum() / 2048
    assert abs(_loss(t) - ref) <= 2.0 ** -23 * ref


@pytest.mark.parametrize("value", [np.inf, -np.inf, 1e25])
def test_infinite_losses(value):
    t = np.ones((40, 192), np.float32)
    t[33, 191] = value
    assert _loss(t) == np.inf


def test_nan_target():
    t = np.ones((40, 192), np.float32)
    t[3, 7] = np.nan
    assert np.isnan(_loss(t))
