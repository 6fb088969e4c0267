"""Steps queued behind one another in the shapes a step can take (two CTAs per
SM, transport's four, shallow water) and with a network, given per-patch
thresholds or hi + lo coarse samples: twelve steps queued at once, and the
same captured and replayed, give the records of a run that is synchronised
after every step.  Grids meant for two CTAs per SM have the patches that the
rule asks for (four per SM for nine fields, one and a half for three)."""
import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import Sim, learned

pytestmark = pytest.mark.gpu


def _nsm():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _grid(kind):
    """Cells per axis: 32-cell kinds with enough patches for half-SM CTAs."""
    if kind in ("half", "half_eps"):
        return 32 * 32, 32 * (4 * _nsm() // 32 + 1)
    if kind == "swe_half":
        return 32 * 16, 32 * (3 * _nsm() // 32 + 1)
    return 256, 192


def _make(kind, stream=None):
    nx, ny = _grid(kind)
    scheme = {"swe_half": "swe", "transport": "transport"}.get(kind, "d2q9")
    P, L = (32, 3) if kind in ("half", "half_eps") else ((32, 4) if kind == "swe_half" else (64, 4))
    y, x = np.mgrid[0:ny, 0:nx]
    noise = 10.0 ** (-3.0 - 4.0 * x / nx) * np.random.default_rng(2).normal(size=(ny, nx))
    w, one = np.sin(2 * np.pi * y / ny) + noise, np.ones((ny, nx))
    f = {"swe": [1.5 + 0.2 * w, 0.1 * w, 0 * one], "transport": [1.0 + 0.1 * w]}.get(scheme, [one, 0.04 * w, 0 * one])
    s = Sim(scheme, "bl53", nx, ny, P, L, 1e-5, prec="f32", store="bf16" if scheme == "d2q9" else "f32", tau=0.7, cfl=0.3,
            velocity=(0.7, 0.6), arena_factor=2.0, stream=stream, coarse_hilo=kind == "hilo")
    if kind == "half_eps":
        learned.set_patch_eps(s, 1e-5 * 10.0 ** np.random.default_rng(3).uniform(-1, 1, s.npatch))
    if kind == "network":
        s.net = learned.Mlp(6 * L, seed=1)
        learned.use_mlp(s, s.net, 1e-7, 1e-3)
    s.init_macro(f)
    if kind == "half":
        assert s.npatch >= 4 * _nsm()
    if kind == "swe_half":
        assert 2 * s.npatch >= 3 * _nsm()
    return s


def _records(s):
    s.sync()
    return [s.record(p) for p in range(s.npatch)]


@pytest.mark.parametrize("kind", ["half", "half_eps", "swe_half", "transport", "network", "hilo"])
def test_queued_and_captured_steps(kind):
    import torch
    ref = _make(kind)
    for _ in range(12):
        ref.step(1)
        ref.sync()
    want = _records(ref)
    st = torch.cuda.Stream()
    a = _make(kind, st)
    a.step(12)
    assert _records(a) == want
    b = _make(kind, st)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        b.step(12)
    g.replay()
    torch.cuda.synchronize()
    assert _records(b) == want
    if kind == "hilo":
        assert np.array_equal(a.coarse_lo(), ref.coarse_lo()) and np.array_equal(b.coarse_lo(), ref.coarse_lo())


def test_per_patch_thresholds_with_two_ctas_per_sm_match_oracle():
    g = _make("half_eps")
    nx, ny = _grid("half_eps")
    y, x = np.mgrid[0:ny, 0:nx]
    noise = 10.0 ** (-3.0 - 4.0 * x / nx) * np.random.default_rng(2).normal(size=(ny, nx))
    o = O.OracleSim("d2q9", "bl53", nx, ny, 32, 3, 1e-5, prec="f32", store="bf16", tau=0.7)
    o.set_patch_eps(1e-5 * 10.0 ** np.random.default_rng(3).uniform(-1, 1, g.npatch))
    o.init_macro([np.ones((ny, nx)), 0.04 * (np.sin(2 * np.pi * y / ny) + noise), np.zeros((ny, nx))])
    for step in range(3):
        for p in range(g.npatch):
            assert g.record(p) == o.record(p), "patch %d differs after %d steps" % (p, step)
        g.step(1)
        o.step(1)
        g.sync()
