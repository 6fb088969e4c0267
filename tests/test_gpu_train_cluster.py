"""Training in one launch: every step equals the gradient of the separate
gradient kernel followed by Adam in FP32, for whole and ragged slices, one
slice to eight, few and many inputs; and batches beyond eight slices, which
keep a launch per minibatch, do as well."""
import numpy as np
import pytest

from paper_2302_09883_gb300 import learned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nin,batch", [(24, 128), (1, 16), (18, 17), (42, 100), (64, 1), (7, 128), (24, 129), (42, 300)])
def test_steps_are_gradient_then_adam(nin, batch):
    import torch
    rng = np.random.default_rng(nin + batch)
    n, epochs, lr = 2 * batch + 1, 3, np.float32(2e-3)
    X = torch.from_numpy(rng.normal(size=(n, nin)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.normal(size=n).astype(np.float32)).cuda()
    m = learned.Mlp(nin, seed=3)
    w = m.weights()
    hist = m.train(X, t, epochs, batch, float(lr), seed=9)
    order = np.random.default_rng(9)
    m1, m2 = np.zeros_like(w), np.zeros_like(w)
    g1, g2 = np.float32(0.9), np.float32(0.999)
    k = 0
    for ep in range(epochs):
        perm = order.permutation(n)[:(n // batch) * batch]
        for b in perm.reshape(-1, batch):
            ref = learned.Mlp(nin, weights=w)
            loss, g = ref.grad(X[torch.from_numpy(b).cuda()], t[torch.from_numpy(b).cuda()])
            ref.close()
            k += 1
            m1 = g1 * m1 + (np.float32(1) - g1) * g
            m2 = g2 * m2 + (np.float32(1) - g2) * g * g
            mh, vh = m1 / (np.float32(1) - g1 ** np.float32(k)), m2 / (np.float32(1) - g2 ** np.float32(k))
            w = w - lr * mh / (np.sqrt(vh) + np.float32(1e-8))
        assert abs(hist[ep] - loss) <= 2e-6 * max(1.0, abs(loss))
    # the bias corrections' power functions may differ in the last bit: 1e-7
    # relative of each of six updates of at most lr
    assert np.max(np.abs(m.weights() - w)) <= 6 * 2e-7 * float(lr) + 4e-7 * np.max(np.abs(w))
