"""3-D labels and features against the oracle where the FP32 decision can go
wrong: one and several fields, grids with a different number of patches per
axis, patches at either end of the labels, values whose squares leave FP32's
range, and patches that are zero or not finite."""
import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import learned

pytestmark = pytest.mark.gpu


def _dense(F, n, P, seed, scale):
    nz, ny, nx = n
    rng = np.random.default_rng(seed)
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx]
    out = np.empty((F,) + n)
    for f in range(F):
        amp = 10.0 ** rng.uniform(-8, -1, (nz // P, ny // P, nx // P))
        amp = amp.repeat(P, 0).repeat(P, 1).repeat(P, 2)
        out[f] = 0.4 + 0.1 * np.sin(2 * np.pi * (x / nx + f * y / ny + z / nz)) + amp * rng.normal(size=n)
    return (scale * out).astype(np.float32)


def _check(d, P, L, delta):
    import torch
    _, nz, ny, nx = d.shape
    feat, lab = learned.features_labels3(torch.from_numpy(d).cuda(), P, L, delta)
    feat, lab = feat.cpu().numpy(), lab.cpu().numpy()
    pid = 0
    for pz in range(nz // P):
        for py in range(ny // P):
            for px in range(nx // P):
                ix = [(p * P + np.arange(P + 1)) % m for p, m in ((pz, nz), (py, ny), (px, nx))]
                v = d.astype(np.float64)[:, ix[0]][:, :, ix[1]][:, :, :, ix[2]]
                fo = O.patch_features(v, "bl53", P, L, prec="f32")
                assert np.max(np.abs(feat[pid] - fo)) <= 2e-6 * max(1.0, np.max(np.abs(fo))), pid
                lo = O.patch_label(v, "bl53", P, L, delta, prec="f32")
                assert abs(lab[pid] - lo) <= 1e-6, (pid, lab[pid], lo)
                pid += 1


@pytest.mark.parametrize("P,n,F,delta,scale", [(16, (16, 32, 48), 19, 1e-5, 1.0), (16, (32, 16, 16), 1, 1e-7, 1.0),
                                               (16, (16, 16, 32), 3, 1e-2, 1.0), (16, (16, 16, 32), 2, 1e-5, 1e-15),
                                               (16, (16, 16, 16), 2, 1e-5, 0.0), (32, (32, 32, 64), 3, 1e-5, 1.0),
                                               (16, (16, 16, 32), 2, 1e-5, 1e16)])
def test_labels3_match_oracle(P, n, F, delta, scale):
    _check(_dense(F, n, P, P + F, scale), P, 3, delta)


def test_non_finite_patch3_takes_the_lowest_label():
    import torch
    d = _dense(2, (16, 16, 32), 16, 1, 1.0)
    d[1, 4, 10, 20] = np.nan
    _, lab = learned.features_labels3(torch.from_numpy(d).cuda(), 16, 3, 1e-4)
    lab = lab.cpu().numpy()
    assert lab[1] == -7.0 and lab[0] > -7.0
