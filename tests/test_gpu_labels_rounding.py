"""2-D labels at bounds near and below the rounding of the FP64 transforms: node
values over fourteen decades, so that the round trip through the transforms
is off by about 2e-16 of the patch's norm, and bounds delta from a tenth of
that on.  The FP64 error decides, with its rounding, as in the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2302_09883_gb300 import learned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,L,F", [(64, 4, 2), (32, 3, 9)])
@pytest.mark.parametrize("delta", [1e-17, 1e-16, 1e-14, 1e-9, 1e-8, 3e-8])
def test_labels_at_tiny_bounds_match_oracle(P, L, F, delta):
    import torch
    rng = np.random.default_rng(P)
    d = rng.choice([-1.0, 1.0], size=(F, P, 2 * P)) * 10.0 ** rng.uniform(-6, 8, size=(F, P, 2 * P))
    d = d.astype(np.float32)
    _, lab = learned.features_labels(torch.from_numpy(d).cuda(), P, L, delta)
    lab = lab.cpu().numpy()
    for px in range(2):
        ix, iy = (px * P + np.arange(P + 1)) % (2 * P), np.arange(P + 1) % P
        lo = O.patch_label(d.astype(np.float64)[:, iy][:, :, ix], "bl53", P, L, delta)
        assert abs(lab[px] - lo) <= 1e-6, (px, lab[px], lo)
        assert delta > 1e-16 or lo == -7.0
