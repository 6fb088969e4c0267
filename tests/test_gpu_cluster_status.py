"""A state that becomes non-finite while a cluster of CTAs steps each patch:
the step that made it so is reported, the steps queued behind it change
nothing, and the records are those of the state before it.  Two populations
of 1.5e308 run towards each other with next to no relaxation (tau 1e6), so
their node's density overflows after two or three steps."""
import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import Sim
from paper_2302_09883_gb300._lib import WcsError

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npx,npy", [(4, 4), (7, 4), (5, 7)])  # clusters of five, five and three
@pytest.mark.parametrize("gap,bad", [(2, 1), (6, 2)])
def test_non_finite_step_is_reported_and_its_input_kept(npx, npy, gap, bad):
    nx, ny = 32 * npx, 32 * npy
    one = np.ones((ny, nx))
    state = np.zeros((9, ny, nx)) + np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    state[1, 40, 41] = state[3, 40, 41 + gap] = 1.5e308
    kw = dict(prec="f64", store="f64", tau=1e6)
    g = Sim("d2q9", "haar", nx, ny, 32, 3, 1e-4, arena_factor=2.0, **kw)
    o = O.OracleSim("d2q9", "haar", nx, ny, 32, 3, 1e-4, **kw)
    for s in (g, o):
        s.init_macro([one, 0 * one, 0 * one])
        s.import_field(-1, state)
    o.step(bad)
    assert np.isfinite(o.export_all()).all()
    g.step(6)
    with pytest.raises(WcsError) as e:
        g.sync()
    assert "E_NAN" in str(e.value) and "at step %d" % bad in str(e.value)
    for p in range(g.npatch):
        assert g.record(p) == o.record(p), p
    o.step(1)
    with np.errstate(all="ignore"):
        assert not np.isfinite(o.export_all()).all()
