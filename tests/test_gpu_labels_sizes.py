"""Labels and features of the register-line kernels against the oracle: the
sizes they are chosen for, one and several fields, patches whose label sits
at either end, and patches so small in value (or not finite) that only the
FP64 decision is left."""
import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import learned

pytestmark = pytest.mark.gpu


def _dense(F, ny, nx, P, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:ny, 0:nx]
    out = np.empty((F, ny, nx))
    for f in range(F):
        amp = 10.0 ** rng.uniform(-9, -1, (ny // P, nx // P)).repeat(P, 0).repeat(P, 1)
        out[f] = 0.4 + 0.1 * np.sin(2 * np.pi * (x / nx + f * y / ny)) + amp * rng.normal(size=(ny, nx))
    return (scale * out).astype(np.float32)


def _nodes(u, P, px, py):
    ny, nx = u.shape[1:]
    ix, iy = (px * P + np.arange(P + 1)) % nx, (py * P + np.arange(P + 1)) % ny
    return u[:, iy][:, :, ix]


@pytest.mark.parametrize("P,L,F,delta,scale", [(64, 4, 9, 1e-5, 1.0), (64, 4, 4, 1e-3, 1.0), (64, 4, 1, 1e-7, 1.0),
                                               (32, 3, 9, 3e-6, 1.0), (32, 3, 1, 1e-2, 1.0), (32, 3, 3, 1e-5, 1e-15),
                                               (64, 4, 2, 1e-5, 0.0)])
def test_register_line_labels_match_oracle(P, L, F, delta, scale):
    import torch
    d = _dense(F, 2 * P, 3 * P, P, seed=P + F, scale=scale)
    feat, lab = learned.features_labels(torch.from_numpy(d).cuda(), P, L, delta)
    feat, lab = feat.cpu().numpy(), lab.cpu().numpy()
    for pid in range(6):
        v = _nodes(d.astype(np.float64), P, pid % 3, pid // 3)
        fo = O.patch_features(v, "bl53", P, L)
        assert np.max(np.abs(feat[pid] - fo)) <= 1e-5 * max(1.0, np.max(np.abs(fo))), pid
        lo = O.patch_label(v, "bl53", P, L, delta)
        assert abs(lab[pid] - lo) <= 1e-6, (pid, lab[pid], lo)


def test_non_finite_patch_takes_the_lowest_label():
    import torch
    d = _dense(2, 64, 128, 64, seed=1)
    d[1, 10, 70] = np.nan
    _, lab = learned.features_labels(torch.from_numpy(d).cuda(), 64, 4, 1e-4)
    lab = lab.cpu().numpy()
    assert lab[1] == -7.0 and lab[0] > -7.0
