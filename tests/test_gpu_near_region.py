"""The immersed-boundary chain of a step waits for the near region only, also on
the steps on which the support box moves by a cell: runs whose body reaches the
box's last cells equal, bit for bit, the same run with the chain behind the whole
window (a re-injection that never triggers)."""
import numpy as np
import pytest

from paper_2408_15115_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# the support box is 18 cells wide and the body reaches its last stencil cell when
# the centre is `slack` past a cell face; vertices lie on the axes


def _run(nx, ny, slack, storage, form, steps):
    from paper_2408_15115_gb300 import turret as T
    radius = 6.0 - 2.0 - 1e-3 - slack
    V, Tr = I.icosphere(4, radius)
    assert np.allclose(np.abs(V).max(0), radius, atol=1e-6)
    shape = (40, ny, nx)
    t = T.Turret(nx, ny, 40, 0.05, 2.0, (0, 0, -1e-4), 0, 0, 1, 2, sponge=4, storage=storage,
                 flags={"no_graph": 1} if form == "no_graph" else None)
    t.set_fields(*I.random_state(shape, u_amp=0.02, rho_amp=0.001, kmax=3, seed=5))
    if form == "whole":
        t.set_reinjection(1, 2, 0, 0)
    # the centre crosses cell faces on every axis, in both directions
    t.load_surface(V, Tr, (8.97, 9.03, 20.02), (0.07, -0.06, -0.05), (0.002, 0.001, 0))
    if form == "batch":
        b = T.Batch([t])
        b.step(steps)
        b.close()
    else:
        t.step(steps)
    s = t.state()
    out = np.concatenate([np.ravel(s[k]) for k in ("r", "v", "w", "F", "T")]), t.populations().cpu().numpy()
    t.close()
    return out


@pytest.mark.parametrize("storage", ["f32", "f16"])
# x: the box fills the axis, or one cell, two or more are left; 64: the x-pair form
# (0.499 and 0.501: a layer around the box, and none)
@pytest.mark.parametrize("nx,ny,slack", [(18, 19, 1e-3), (20, 33, 1e-3), (64, 18, 1e-3), (18, 20, 0.499), (19, 18, 0.501)])
def test_chain_behind_the_near_region_alone(nx, ny, slack, storage):
    steps = 43
    want = _run(nx, ny, slack, storage, "whole", steps)
    assert np.floor(want[0][2]) < 20  # faces were crossed
    for form in ("graph", "no_graph", "batch"):
        got = _run(nx, ny, slack, storage, form, steps)
        assert np.array_equal(got[0], want[0]), form
        assert np.array_equal(got[1], want[1]), form
