"""Steps launched behind one another: runs on two streams in turn, statistics
queued between steps, and steps captured into a graph and replayed once give
the records of a run that is synchronised after every step."""
import numpy as np
import pytest

from paper_2302_09883_gb300 import Sim, inputs

pytestmark = pytest.mark.gpu

KINDS = [("d2q9", "bl53", 192, 128, 64, 4, "f32", "bf16"), ("d2q9", "haar", 128, 128, 32, 3, "f64", "f64"),
         ("euler2d", "bl53", 128, 192, 64, 4, "f32", "i8")]


def _make(kind, stream=None):
    scheme, wavelet, nx, ny, P, L, prec, store = kind
    y, x = np.mgrid[0:ny, 0:nx]
    w = np.sin(2 * np.pi * y / ny) + 1e-3 * np.random.default_rng(2).normal(size=(ny, nx))
    one = np.ones((ny, nx))
    f = [one, 0.04 * w, 0 * one] if scheme == "d2q9" else [one + 0.1 * w, 0.2 * w, 0 * one, one]
    s = Sim(scheme, wavelet, nx, ny, P, L, 1e-5, prec=prec, store=store, tau=0.7, cfl=0.3, arena_factor=2.0, stream=stream)
    s.init_macro(f)
    return s


def _records(s):
    s.sync()
    return [s.record(p) for p in range(s.npatch)]


@pytest.mark.parametrize("kind", KINDS)
def test_streams_stats_and_capture(kind):
    import torch
    ref = _make(kind)
    for _ in range(12):
        ref.step(1)
        ref.sync()
    want, mass = _records(ref), ref.stats()["mass"]
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    a, b = _make(kind, sa), _make(kind, sb)
    for k in range(12):
        a.step(1)
        b.step(1)
        a.stats_enqueue(k % 4)
        if k % 4 == 3:
            for q in range(4):
                st = a.stats_collect(q)
    assert _records(a) == want and _records(b) == want and st["mass"] == mass
    c = _make(kind, sa)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=sa):
        c.step(12)
    g.replay()
    torch.cuda.synchronize()
    assert _records(c) == want
