"""The lines between the codec's three ways to take survivors (a warp per word,
a thread per survivor, whole rows): patches with none to many isolated spikes,
so that their numbers of stored words lie on both sides of both lines (64
words, a third of all).  Records byte-identical to the oracle's over steps."""
import struct

import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import Sim

pytestmark = pytest.mark.gpu

SPIKES = (0, 1, 2, 3, 4, 6, 8, 12, 16, 24, 48, 96)


def _state(P, scheme):
    nx, ny = P * len(SPIKES), P
    rng = np.random.default_rng(P)
    bump = np.zeros((ny, nx))
    for k, n in enumerate(SPIKES):
        at = rng.choice(P * P, size=n, replace=False)
        bump[at // P, k * P + at % P] = rng.uniform(0.01, 0.03, n)
    one = np.ones((ny, nx))
    if scheme == "d2q9":
        return nx, ny, [one + bump, 0.02 * one, 0 * one]
    return nx, ny, [1.5 + bump, 0.1 * one, 0 * one] if scheme == "swe" else [one + bump, 0.2 * one, 0 * one, one]


def _words(record):
    F = struct.unpack_from("<I", record, 8)[0]
    return sum(struct.unpack_from("<4I", record, 16 + 16 * f)[1] for f in range(F))


@pytest.mark.parametrize("scheme,wavelet,prec,store,P,L", [("d2q9", "bl53", "f32", "bf16", 64, 4), ("d2q9", "bl53", "f32", "i8", 64, 4),
                                                           ("d2q9", "bl53", "f32", "f32", 32, 3), ("d2q9", "haar", "f64", "f64", 32, 3),
                                                           ("euler2d", "bl53", "f32", "i8", 64, 4), ("swe", "bl53", "f64", "f64", 32, 3)])
def test_records_on_both_sides_of_each_line(scheme, wavelet, prec, store, P, L):
    nx, ny, f = _state(P, scheme)
    kw = dict(prec=prec, store=store, tau=0.8, cfl=0.2)
    g = Sim(scheme, wavelet, nx, ny, P, L, 1e-4, arena_factor=2.0, **kw)
    o = O.OracleSim(scheme, wavelet, nx, ny, P, L, 1e-4, **kw)
    g.init_macro(f)
    o.init_macro(f)
    E, F = P + (wavelet == "bl53"), g.F
    nw = E * (P // 32) + ((E + 31) // 32 if E > P else 0)
    words = []
    for step in range(4):
        g.sync()
        for p in range(g.npatch):
            r = o.record(p)
            words.append(_words(r))
            assert g.record(p) == r, "patch %d differs after %d steps" % (p, step)
        g.step(1)
        o.step(1)
    some, dense = 64, F * nw // 3
    assert any(0 < w <= some for w in words) and any(w >= dense for w in words)
    assert dense <= some or any(some < w < dense for w in words)
