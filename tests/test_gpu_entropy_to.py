"""The entry that asks for memory once the coded size is known: the check that
the coded state decodes back has ended before the caller's memory is asked
for (the stream has nothing left to do), so that a state that does not decode
back leaves that memory as it is."""
import ctypes as C

import numpy as np
import pytest

from paper_2302_09883_gb300 import Sim, _lib as B

pytestmark = pytest.mark.gpu


def _state(nx, ny):
    # every detail kept, in FP32: records of some 150 KB, whose decode takes long beside a host call
    y, x = np.mgrid[0:ny, 0:nx]
    f = [np.ones((ny, nx)), 0.04 * np.sin(2 * np.pi * y / ny) + 1e-3 * np.random.default_rng(1).normal(size=(ny, nx)),
         np.zeros((ny, nx))]
    g = Sim("d2q9", "bl53", nx, ny, 64, 4, 0.0, prec="f32", store="f32", tau=0.6, arena_factor=2.0)
    g.init_macro(f)
    return g


def test_memory_is_asked_for_behind_the_check():
    import torch
    g = _state(512, 256)
    buf, seen = np.zeros(9 * 4 * 512 * 256 * 2, np.uint8), []

    def alloc(_, n):
        seen.append((torch.cuda.current_stream().query(), n))
        return buf.ctypes.data

    n = C.c_int64()
    B.check(B.lib().wcs_entropy_code_to(g.h, B.ALLOC(alloc), None, C.byref(n)), g.h)
    assert seen == [(True, n.value)]
    assert buf[:n.value].tobytes() == g.entropy_code()


def test_temporary_memory_is_bounded():
    # what is held while the caller is asked for memory: 1.5 bytes for each of
    # the records, the coded state, some words per record and table
    import torch
    g = _state(1024, 1024)
    g.entropy_code()  # the kernels are loaded
    torch.cuda.synchronize()
    before, held = torch.cuda.mem_get_info()[0], []
    live, n = g.stats()["live_bytes"], C.c_int64()

    def alloc(_, k):
        held.append(before - torch.cuda.mem_get_info()[0])
        return None

    B.check(B.lib().wcs_entropy_code_to(g.h, B.ALLOC(alloc), None, C.byref(n)), g.h)
    granule = 2 << 20  # device memory is handed out in pieces of 2 MiB
    assert live > 36 << 20
    assert held[0] <= 1.5 * live + n.value + 128 * g.npatch + 65536 + 2 * granule
