"""The entropy stage where its kernels can go wrong: records of the smallest
size, one patch and more patches than lanes of a launch, a state of equal
bytes almost throughout, every detail kept; and the size asked for alone, a
buffer that is too small, and the same bytes from both entries."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import Sim, _lib as B, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme,store,P,L,nx,ny,eps", [("transport", "f32", 64, 5, 64, 64, 1e-1),
                                                        ("transport", "f32", 64, 1, 128, 64, 0.0),
                                                        ("d2q9", "bf16", 32, 3, 2080, 1216, 1e-4),
                                                        ("d2q9", "f32", 32, 3, 96, 32, 0.0)])
def test_coded_state_matches_oracle(scheme, store, P, L, nx, ny, eps):
    kw = dict(tau=0.6) if scheme == "d2q9" else dict(velocity=(0.9, 0.9), cfl=0.45)
    y, x = np.mgrid[0:ny, 0:nx]
    w = np.sin(2 * np.pi * y / ny) + 1e-3 * np.random.default_rng(1).normal(size=(ny, nx)) * (x < nx // 2)
    f = [1.0 + 0.1 * w] if scheme == "transport" else [np.ones((ny, nx)), 0.04 * w, np.zeros((ny, nx))]
    g = Sim(scheme, "bl53", nx, ny, P, L, eps, prec="f32", store=store, arena_factor=2.0, **kw)
    o = O.OracleSim(scheme, "bl53", nx, ny, P, L, eps, prec="f32", store=store, **kw)
    g.init_macro(f)
    o.init_macro(f)
    code = g.entropy_code()
    assert code == o.entropy_code()
    n = C.c_int64()
    assert B.lib().wcs_entropy_code(g.h, None, 0, C.byref(n)) == 0 and n.value == len(code)
    small = np.zeros(len(code) - 1, np.uint8)
    assert B.lib().wcs_entropy_code(g.h, small.ctypes.data, small.size, C.byref(n)) == 1 and n.value == len(code)
    assert not small.any()
    buf = np.zeros(len(code), np.uint8)
    assert B.lib().wcs_entropy_code(g.h, buf.ctypes.data, buf.size, C.byref(n)) == 0 and buf.tobytes() == code
