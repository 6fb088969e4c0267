"""The codec's paths by how many mask words a patch stores: none, a few (the
word list; at most 32 words of a field come with its presence bits), many
(whole rows), all (eps = 0).  Records byte-identical to the oracle of the
same precision, over several steps so that own decode, ghost decode and
writer all run at each density."""
import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import Sim, inputs

pytestmark = pytest.mark.gpu


def _fields(scheme, nx, ny, periodic, seed):
    rng = np.random.default_rng(seed)
    gx, gy = nx + (not periodic), ny + (not periodic)
    y, x = np.mgrid[0:gy, 0:gx]
    # noise whose amplitude falls from left to right: every density in one grid
    noise = 10.0 ** (-3.0 - 4.0 * x / gx) * rng.normal(size=(gy, gx))
    wave = np.sin(2 * np.pi * y / gy)
    if scheme == "d2q9":
        return [np.ones((gy, gx)), 0.04 * wave + noise, np.zeros((gy, gx))]
    if scheme == "euler2d":
        one = np.ones((gy, gx))
        return [one + 0.1 * wave + noise, 0.3 * wave, 0.1 * one, one + noise]
    if scheme == "transport":
        return [1.0 + 0.5 * wave + noise]
    return [1.5 + 0.2 * wave + noise, 0.1 * wave, np.zeros((gy, gx))]


@pytest.mark.parametrize("eps", [0.0, 1e-6, 3e-5, 1e-3])
@pytest.mark.parametrize("scheme,prec,store,P,L,periodic", [
    ("d2q9", "f32", "bf16", 64, 4, True), ("d2q9", "f32", "f32", 64, 4, True), ("d2q9", "f32", "i8", 64, 4, True),
    ("d2q9", "f32", "bf16", 32, 3, True), ("d2q9", "f32", "f32", 32, 3, True), ("d2q9", "f64", "f64", 32, 3, True),
    ("euler2d", "f32", "i8", 64, 4, False), ("euler2d", "f32", "bf16", 64, 4, True), ("euler2d", "f64", "f64", 32, 3, False),
    ("transport", "f32", "f32", 64, 1, False), ("transport", "f32", "f32", 64, 5, True),
    ("swe", "f32", "f32", 64, 4, False), ("swe", "f32", "f32", 32, 4, True), ("swe", "f64", "f64", 32, 3, False)])
def test_records_at_every_density(scheme, prec, store, P, L, periodic, eps):
    nx, ny = 3 * P, 2 * P
    per = (periodic, periodic)
    kw = dict(prec=prec, store=store, periodic=per, tau=0.6, cfl=0.3)
    if scheme == "transport":
        kw.update(velocity=(0.9, 0.7))
    g = Sim(scheme, "bl53", nx, ny, P, L, eps, arena_factor=2.0, **kw)
    o = O.OracleSim(scheme, "bl53", nx, ny, P, L, eps, **kw)
    f = _fields(scheme, nx, ny, periodic, seed=7)
    g.init_macro(f)
    o.init_macro(f)
    for step in range(4):
        g.sync()
        for p in range(g.npatch):
            assert g.record(p) == o.record(p), "patch %d differs after %d steps" % (p, step)
        g.step(1)
        o.step(1)
