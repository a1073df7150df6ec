"""The warm-start network at the batch sizes where its kernels change: a few rows (blocks
of 32, tiles of 128), the first batch of each column tile of the products (on 152 SMs 32
columns up to 2 432 rows, 64 up to 4 864, 128 up to 9 728, 256 beyond), and output arrays
that are not 16-byte aligned. References and tolerances of test_gpu_mlp.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as om  # noqa: E402

pytestmark = pytest.mark.gpu

NIN = om.DIMS[0][0]
K_GRAD = 4.0


def _setup(fil, B):
    rng = np.random.default_rng(B)
    p = np.concatenate([np.concatenate([rng.standard_normal(i * o) * np.sqrt(2.0 / i),
                                        0.1 * rng.standard_normal(o)])
                        for i, o in om.DIMS]).astype(np.float32)
    norm = [rng.standard_normal(NIN).astype(np.float32), rng.uniform(0.5, 2, NIN).astype(np.float32),
            rng.standard_normal(192).astype(np.float32), rng.uniform(0.5, 2, 192).astype(np.float32)]
    m = fil.fil_mlp_create(B)
    fil.fil_mlp_set_params(m, p)
    fil.fil_mlp_set_norm(m, *norm)
    x = (norm[0] + norm[1] * rng.standard_normal((B, NIN))).astype(np.float32)
    t = (norm[2] + norm[3] * rng.standard_normal((B, 192))).astype(np.float32)
    return m, p, norm, x, t


def _out(n, offset):
    """n floats, `offset` floats past a 16-byte boundary, between guard values."""
    buf = torch.full((n + 8,), 7.5, device="cuda")
    assert buf.data_ptr() % 16 == 0
    return buf, buf[offset:offset + n]


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("B", [1, 31, 33])
def test_forward(B, offset):
    from paper_1903_12609_gb300 import fil
    m, p, norm, x, _ = _setup(fil, B)
    buf, y = _out(B * 192, offset)
    fil.fil_mlp_forward(m, torch.from_numpy(x).cuda(), y, B)
    fil.fil_mlp_destroy(m)
    ref, _ = om.forward(p, x, norm)
    scale = np.abs(ref - norm[2]).max()
    np.testing.assert_allclose(y.cpu().numpy().reshape(B, 192), ref, rtol=0, atol=2e-3 * scale)
    assert bool((buf[:offset] == 7.5).all()) and bool((buf[offset + B * 192:] == 7.5).all())


@pytest.mark.parametrize("B,offset", [(1, 0), (31, 3), (33, 0), (65, 1), (2433, 0), (4865, 0)])
def test_gradients(B, offset):
    from paper_1903_12609_gb300 import fil
    m, p, norm, x, t = _setup(fil, B)
    buf, g = _out(om.NPARAM, offset)
    loss = fil.fil_mlp_gradients(m, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), B, g)
    fil.fil_mlp_destroy(m)
    ref_loss, ref = om.loss_and_grad(p, x, t, norm)
    mag = om.grad_magnitudes(p, x, t, norm)
    assert abs(loss - ref_loss) <= 1e-4 * ref_loss
    g = g.cpu().numpy()
    assert np.all(np.abs(g - ref) <= K_GRAD * 2.0 ** -8 * mag + 1e-30)
    off = 0
    for i, o in om.DIMS:
        for n in (i * o, o):
            assert np.linalg.norm((g - ref)[off:off + n]) <= 1e-2 * np.linalg.norm(ref[off:off + n])
            off += n
    assert bool((buf[:offset] == 7.5).all()) and bool((buf[offset + om.NPARAM:] == 7.5).all())


@pytest.mark.parametrize("B", [2432, 2433, 4865, 9729])
def test_rows_do_not_depend_on_the_tiles(B):
    """Every tile width adds a row's K blocks in the same order: the outputs of a batch are
    bit for bit those of its rows in batches of 1 280 (32-column tiles)."""
    from paper_1903_12609_gb300 import fil
    m, _, _, x, _ = _setup(fil, B)
    x, y = torch.from_numpy(x).cuda(), torch.full((B, 192), float("nan"), device="cuda")
    fil.fil_mlp_forward(m, x, y, B)
    for i in range(0, B, 1280):
        n = min(1280, B - i)
        part = torch.full((n, 192), float("nan"), device="cuda")
        fil.fil_mlp_forward(m, x[i:i + n], part, n)
        assert torch.equal(y[i:i + n], part)
    fil.fil_mlp_destroy(m)


def test_gradient_of_the_widest_tiles():
    """10 240 rows against the mean over eight batches of 1 280: dY / B has the same BF16
    roundings (B differs by a power of two), so only the sums over the batch differ, by
    the roundings of B / 16 accumulation steps, 2^-23 each of sums of the result's size."""
    from paper_1903_12609_gb300 import fil
    B = 10240
    m, _, _, x, t = _setup(fil, B)
    x, t = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    g, part = torch.empty(om.NPARAM, device="cuda"), torch.empty(om.NPARAM, device="cuda")
    loss = fil.fil_mlp_gradients(m, x, t, B, g)
    mean, lmean = torch.zeros(om.NPARAM, dtype=torch.float64, device="cuda"), 0.0
    for i in range(0, B, 1280):
        lmean += fil.fil_mlp_gradients(m, x[i:i + 1280], t[i:i + 1280], 1280, part) / 8
        mean += part.double() / 8
    fil.fil_mlp_destroy(m)
    assert abs(loss - lmean) <= 2.0 ** -22 * lmean
    off = 0
    for i, o in om.DIMS:
        for n in (i * o, o):
            d = (g.double() - mean)[off:off + n]
            assert float(d.norm()) <= B / 16 * 2.0 ** -23 * float(mean[off:off + n].norm())
            off += n


@pytest.mark.parametrize("M,N,K", [(19 * 128 + 1, 256, 128), (38 * 128 + 1, 288, 576),
                                   (76 * 128 + 1, 192, 64), (152 * 128 + 1, 288, 576)])
def test_product_tiles(M, N, K):
    """Tiles of 64 to 256 columns with a remainder in rows and columns."""
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(N + K)
    A = om.bf16_round(rng.standard_normal((M, K)).astype(np.float32))
    B = om.bf16_round(rng.standard_normal((N, K)).astype(np.float32))
    dev = [torch.from_numpy(om.bf16_bits(v).view(np.int16)).cuda() for v in (A, B)]
    C = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    fil.fil_tc_gemm_bf16(dev[0], K, dev[1], K, C, N, M, N, K)
    bound = 2.0 ** -22 * K * (np.abs(A).max(axis=1)[:, None] * np.abs(B).max(axis=1)[None, :])
    assert np.all(np.abs(C.cpu().numpy() - A @ B.T) <= bound)
