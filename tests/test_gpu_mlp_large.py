"""The warm-start network on batches of more than 65 535 x 32 rows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as om  # noqa: E402

pytestmark = pytest.mark.gpu

NIN = om.DIMS[0][0]
ROWS = 65535 * 32 + 17


def _network(fil, rng, rows):
    m = fil.fil_mlp_create(rows)
    p = np.concatenate([np.concatenate([rng.standard_normal(i * o) * np.sqrt(2.0 / i),
                                        0.1 * rng.standard_normal(o)]) for i, o in om.DIMS])
    fil.fil_mlp_set_params(m, p.astype(np.float32))
    fil.fil_mlp_set_norm(m, *(np.full(n, v, np.float32) for n, v in
                              ((NIN, 0.0), (NIN, 1.0), (192, 0.0), (192, 1.0))))
    return m


def test_rows_past_the_second_grid_dimension():
    """Rows repeat a block of 4096, so that the outputs repeat bit for bit, and the
    loss and gradient are those of the block with each row weighted by how often it
    occurs. Bounds: the block's outputs and loss differ by the tiles' widths only
    (2e-3 of the scale and 1e-4, as in test_gpu_mlp.py); a weight gradient sums K rows
    in K / 16 steps of FP32, and dY / B rounds to BF16 anew: (K / 16) 2^-23 + 2^-7 of
    its norm."""
    from paper_1903_12609_gb300 import fil
    rng = np.random.default_rng(2)
    block = 4096
    xb = torch.from_numpy(rng.standard_normal((block, NIN)).astype(np.float32)).cuda()
    tb = torch.from_numpy(rng.standard_normal((block, 192)).astype(np.float32)).cuda()
    idx = torch.arange(ROWS, device="cuda") % block
    m = _network(fil, rng, ROWS)
    yb = torch.empty(block, 192, device="cuda")
    gb, g = torch.empty(om.NPARAM, device="cuda"), torch.empty(om.NPARAM, device="cuda")
    fil.fil_mlp_forward(m, xb, yb, block)
    lb = fil.fil_mlp_gradients(m, xb, tb, block, gb)
    x, y = xb[idx], torch.empty(ROWS, 192, device="cuda")
    fil.fil_mlp_forward(m, x, y, ROWS)
    assert torch.equal(y, y[:block][idx])
    assert float((y[:block] - yb).abs().max()) <= 2e-3 * float(yb.abs().max())
    loss = fil.fil_mlp_gradients(m, x, tb[idx], ROWS, g)
    fil.fil_mlp_destroy(m)
    # whole blocks, and ROWS % block rows once more: that share of the weight is uneven
    slack = (ROWS % block) / ROWS
    assert abs(loss - lb) <= (1e-4 + 2 * slack) * lb
    assert float((g - gb).norm()) <= (ROWS / 16 * 2.0 ** -23 + 2.0 ** -7 + 2 * slack) * float(gb.norm())
