"""The drag-model J0 solve of one FP64 system in blocks of 16 band rows, at the
edges: one segment (3 rows), the last block's remainder 1 and 15 (14 and 19
segments), a filament of many blocks, the most filaments that solve so (two for
each SM) and one more, which solve row by row; each also in place.

Tolerance: both ways solve with backward-stable factors of J0, so the error is
at most n cond(J0) eps relative to the solution's norm (n unknowns), and the
oracle's dense LU obeys the same bound: 2 n cond eps.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import filament as fo  # noqa: E402
from paper_1903_12609_gb300.inputs import random_frames  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("segs", [[1], [2, 1, 3], [14, 1, 19], [150], "two per SM", "one more"])
def test_solve_matches_the_dense_oracle(segs, in_place):
    from paper_1903_12609_gb300 import fil
    if isinstance(segs, str):
        m = 2 * torch.cuda.get_device_properties(0).multi_processor_count + (segs == "one more")
        segs = ([4, 1, 2] * m)[:m]
    rng = np.random.default_rng(sum(segs))
    lay = fo.Layout(segs)
    p = fo.Params(a=1.0, eta=1.0, dL=2.2, KB=2.0, KT=1.5, dt=0.1, tol=1e-10, max_iter=60)
    base = 400.0 * np.arange(3 * len(segs), dtype=float).reshape(-1, 3)
    t, mu = random_frames(rng, len(segs))
    st = fo.initial_state(lay, p, base, t, mu, 0.05 * rng.standard_normal((lay.S, 3)))
    st.lam = 0.1 * rng.standard_normal((lay.n_lam, 3))
    b = rng.standard_normal(6 * lay.S)
    with fil.Filaments(segs, a=p.a, eta=p.eta, dL=p.dL, KB=p.KB, KT=p.KT, dt=p.dt, tol=p.tol,
                       max_iter=p.max_iter) as m:
        m.set_state(st.Y, st.q, None, st.u, st.lam if lay.n_lam else None)
        m.broyden_begin()
        X0 = np.zeros(6 * lay.S)
        m.get_iterate(X0, None)
        x = torch.tensor(b, device="cuda")
        m.j0_solve(x if in_place else x.clone(), x)
        x = x.cpu().numpy()
    for B, o in zip(fo.jacobian0(lay, p, st, X0), lay.off_X):
        n = B.shape[0]
        ref = np.linalg.solve(B, b[o:o + n])
        tol = 2 * n * np.linalg.cond(B) * np.finfo(float).eps
        err = np.linalg.norm(x[o:o + n] - ref)
        assert err <= tol * np.linalg.norm(ref), (n, err / np.linalg.norm(ref), tol)
        assert tol < 1e-3
