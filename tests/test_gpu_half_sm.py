"""Steps with two CTAs per SM (32-cell patches on grids of many patches): the
records of every patch against the oracle, for each scheme, precision and
storage that takes them, from dense to smooth patches within one grid and
with every detail kept."""
import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import Sim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [0.0, 1e-6, 1e-4])
@pytest.mark.parametrize("scheme,prec,store,L,periodic", [("d2q9", "f32", "bf16", 3, True), ("d2q9", "f32", "f32", 3, True),
                                                          ("swe", "f32", "f32", 4, False), ("swe", "f64", "f64", 3, True)])
def test_steps_of_many_small_patches_match_oracle(scheme, prec, store, L, periodic, eps):
    nx, ny, P = 32 * 22, 32 * 28, 32  # 616 patches
    gx, gy = nx + (not periodic), ny + (not periodic)
    rng = np.random.default_rng(L)
    y, x = np.mgrid[0:gy, 0:gx]
    noise = 10.0 ** (-3.0 - 4.0 * x / gx) * rng.normal(size=(gy, gx))
    wave = np.sin(2 * np.pi * y / gy)
    f = [np.ones((gy, gx)), 0.04 * wave + noise, np.zeros((gy, gx))]
    if scheme == "swe":
        f = [1.5 + 0.2 * wave + noise, 0.1 * wave, np.zeros((gy, gx))]
    kw = dict(prec=prec, store=store, periodic=(periodic, periodic), tau=0.6, cfl=0.3)
    g = Sim(scheme, "bl53", nx, ny, P, L, eps, arena_factor=2.0, **kw)
    o = O.OracleSim(scheme, "bl53", nx, ny, P, L, eps, **kw)
    g.init_macro(f)
    o.init_macro(f)
    for step in range(2):
        g.step(1)
        o.step(1)
        g.sync()
        for p in range(g.npatch):
            assert g.record(p) == o.record(p), "patch %d differs after %d steps" % (p, step + 1)
