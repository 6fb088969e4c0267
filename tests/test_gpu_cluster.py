"""Patches shared by a cluster of CTAs (small FP64 Haar grids): the records of
every step equal the oracle's for grids that take clusters of five, of three
and none, at densities from no detail to every detail; a NaN in one patch is
reported as without clusters."""
import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import Sim, _lib, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npx,npy", [(1, 1), (4, 4), (7, 4), (5, 7), (8, 8)])
@pytest.mark.parametrize("eps", [0.0, 1e-4, 1e-2])
def test_records_match_oracle(npx, npy, eps):
    nx, ny = 32 * npx, 32 * npy
    y, x = np.mgrid[0:ny, 0:nx]
    rng = np.random.default_rng(3)
    noise = 10.0 ** (-2.0 - 5.0 * x / nx) * rng.normal(size=(ny, nx))
    f = [1.0 + 0.1 * np.exp(-((x - nx / 2) ** 2 + (y - ny / 2) ** 2) / 128.0), 0.03 * np.sin(2 * np.pi * y / ny) + noise,
         np.zeros((ny, nx))]
    g = Sim("d2q9", "haar", nx, ny, 32, 3, eps, prec="f64", store="f64", tau=0.8, arena_factor=2.0)
    o = O.OracleSim("d2q9", "haar", nx, ny, 32, 3, eps, prec="f64", store="f64", tau=0.8)
    g.init_macro(f)
    o.init_macro(f)
    for step in range(4):
        g.sync()
        for p in range(g.npatch):
            assert g.record(p) == o.record(p), "patch %d differs after %d steps" % (p, step)
        g.step(1)
        o.step(1)
    assert np.array_equal(g.export_field(-1), o.export_all())


def test_nan_is_reported_and_the_state_kept():
    f = inputs.gaussian_bump(128)
    g = Sim("d2q9", "haar", 128, 128, 32, 3, 1e-4, prec="f64", store="f64", tau=0.8)
    f[0][40, 70] = np.nan
    with pytest.raises(_lib.WcsError):
        g.init_macro(f)
        g.step(3)
        g.sync()
    assert g.stats()["status"] & 2


def test_overflowing_arena_is_run_again():
    # noise that grows past the arena of a smooth start: automatic arenas
    f = inputs.gaussian_bump(128, sigma=3.0)
    g = Sim("d2q9", "haar", 128, 128, 32, 3, 1e-9, prec="f64", store="f64", tau=0.8)
    o = O.OracleSim("d2q9", "haar", 128, 128, 32, 3, 1e-9, prec="f64", store="f64", tau=0.8)
    g.init_macro(f)
    o.init_macro(f)
    g.step(30)
    o.step(30)
    g.sync()
    for p in range(g.npatch):
        assert g.record(p) == o.record(p)
