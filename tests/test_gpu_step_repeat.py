"""An iteration whose evaluation fails (here: not finite, from a load of NaN) leaves the
step as it was: with the load put right, fil_broyden_step goes on through the same
iterates, bit for bit, as a step that was never disturbed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _iterates(fil, precision, model, graph, fail_at):
    n, m = 20, 3
    rng = np.random.default_rng(4)
    base = 30.0 * np.arange(m)[:, None] * np.array([1.0, 0.3, 0.0])
    t = rng.standard_normal((m, 3))
    t /= np.linalg.norm(t, axis=1, keepdims=True)
    mu = np.cross(t, [0.3, 0.5, 0.8])
    mu /= np.linalg.norm(mu, axis=1, keepdims=True)
    load = np.tile([0.0, 0.0, -10.0], (m * n, 1))
    bad = load.copy()
    bad[7, 1] = np.nan
    seen, X = [], np.empty(6 * n * m)
    with fil.Filaments([n] * m, KB=200.0, KT=200.0, dt=0.02, tol=1e-9, max_iter=60,
                       precision=precision, j0_model=model) as c:
        c.set_external(load)
        if graph:
            c.set_graph(True)
        c.init_straight(base, t, mu, 1e-2 * rng.standard_normal((m * n, 3)))
        c.broyden_begin()
        done, k = False, 0
        while not done:
            if k == fail_at:
                c.set_external(bad)
                with pytest.raises(fil.FilError) as e:
                    c.broyden_step()
                assert e.value.status == fil.FIL_ENAN
                c.set_external(load)
            done, _ = c.broyden_step()
            c.get_iterate(X)
            seen.append(X.copy())
            k += 1
    return seen


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("precision,model", [("FIL_FP64", "FIL_J0_DRAG"),
                                             ("FIL_MIXED", "FIL_J0_FILAMENT_RPY")])
def test_failed_evaluation_leaves_the_step(precision, model, graph):
    from paper_1903_12609_gb300 import fil
    a = _iterates(fil, getattr(fil, precision), getattr(fil, model), graph, None)
    b = _iterates(fil, getattr(fil, precision), getattr(fil, model), graph, 2)
    assert len(a) == len(b) and len(a) > 3
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
