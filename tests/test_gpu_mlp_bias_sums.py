"""The last layer's bias gradient of the warm-start network is the sum over the batch of
dY = (y - t) / B, whose FP32 terms follow from the outputs when the normalisation is the
identity."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as om  # noqa: E402

pytestmark = pytest.mark.gpu

NIN = om.DIMS[0][0]


@pytest.mark.parametrize("B", [33, 1024, 10240])
def test_sum_of_the_output_errors(B):
    """Against the FP64 sum of the same terms. A compensated sum leaves a rounding of the
    result and one of each partial sum of 32, together sqrt(2) 2^-24 of the norm at most;
    plain sums over the parts round once for each."""
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(B)
    p = np.concatenate([np.concatenate([rng.standard_normal(i * o) * np.sqrt(2.0 / i),
                                        0.1 * rng.standard_normal(o)]) for i, o in om.DIMS])
    m = fil.fil_mlp_create(B)
    fil.fil_mlp_set_params(m, p.astype(np.float32))
    fil.fil_mlp_set_norm(m, *(np.full(n, v, np.float32) for n, v in
                              ((NIN, 0.0), (NIN, 1.0), (192, 0.0), (192, 1.0))))
    x = torch.from_numpy(rng.standard_normal((B, NIN)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.standard_normal((B, 192)).astype(np.float32)).cuda()
    y, g = torch.empty(B, 192, device="cuda"), torch.empty(om.NPARAM, device="cuda")
    fil.fil_mlp_forward(m, x, y, B)
    fil.fil_mlp_gradients(m, x, t, B, g)
    fil.fil_mlp_destroy(m)
    terms = (y - t) * torch.tensor(1.0 / B, dtype=torch.float32, device="cuda")
    ref = terms.double().sum(0)
    err = float((g[-192:].double() - ref).norm() / ref.norm())
    print("bias sum error", B, err)
    assert err <= 2.0 ** -23.5
