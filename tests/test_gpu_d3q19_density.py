"""The 3-D codec by how much a patch stores: nothing but coarse samples,
a few words, every word (eps = 0), on ragged boxes where a CTA takes several
patches.  Records byte-identical to the FP32 oracle over several steps."""
import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import Sim3, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [0.0, 1e-6, 1e-4])
@pytest.mark.parametrize("P,store,box", [(16, "f32", (48, 16, 32)), (16, "bf16", (32, 48, 16)), (32, "f32", (64, 32, 32)),
                                         (32, "bf16", (32, 64, 64))])
def test_records3_at_every_density(P, store, box, eps):
    nx, ny, nz = box
    f = inputs.shear_wave_3d(nx, ny, nz, u0=0.03, axis=1, seed=3)
    x = np.arange(nx)[None, None, :]
    rng = np.random.default_rng(5)
    f[1] = f[1] + 10.0 ** (-3.0 - 5.0 * x / nx) * rng.normal(size=f[1].shape)  # every density in one box
    g = Sim3(nx, ny, nz, P, 3, eps, store=store, tau=0.7, arena_factor=2.0)
    o = O.OracleSim3("bl53", nx, ny, nz, P, 3, eps, prec="f32", store=store, tau=0.7)
    g.init_macro(f)
    o.init_macro(f)
    for step in range(3):
        g.sync()
        for p in range(g.npatch):
            assert g.record(p) == o.record(p), "patch %d differs after %d steps" % (p, step)
        g.step(1)
        o.step(1)
