"""The bounds with which the 2-D labels take a decision from FP32 (no GPU): ERR,
the rounding of the FP32 inverse transform against the 2-norm of what goes in,
and ROUND, that of both FP64 transforms against the patch's norm, recomputed
from the lifting steps as matrices; and the FP32 transform, step by step in
numpy, stays far below the first."""
import os
import re

import numpy as np
import pytest

import oracle as O

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_09883_gb300", "csrc", "mlp.cu")


def _norm(m):
    return float(np.linalg.norm(m, 2)) if m.size else 0.0


def _steps(P, L, inverse):
    """Lifting steps (increment, its first half, nodes changed) of one line."""
    out = []
    for lev in reversed(range(L)):
        st = 1 << lev
        K = P // st // 2
        alpha = [0.5 if k in (0, K - 1) else 0.25 for k in range(K)]
        up, half, pr = (np.zeros((P + 1, P + 1)) for _ in range(3))
        for k in range(1, K):
            up[2 * k * st, (2 * k - 1) * st] = half[2 * k * st, (2 * k - 1) * st] = -alpha[k - 1]
            up[2 * k * st, (2 * k + 1) * st] = -alpha[k]
        for k in range(K):
            pr[(2 * k + 1) * st, [2 * k * st, (2 * k + 2) * st]] = 0.5
        out += [(up, half, [2 * k * st for k in range(1, K)]), (pr, None, [(2 * k + 1) * st for k in range(K)])]
    return out if inverse else [(-u, None if h is None else -h, c) for u, h, c in reversed(out)]


def _line(P, L, inverse, unit):
    """Matrix of the line transform, and its rounding against a unit vector:
    an update rounds both of its products' sums, a predict its sum and result."""
    steps, eye = _steps(P, L, inverse), np.eye(P + 1)
    pre, post, r = [eye], [], eye
    for u, _, _ in steps:
        pre.append((eye + u) @ pre[-1])
    for u, _, _ in reversed(steps):
        post.insert(0, r)
        r = r @ (eye + u)
    err = 0.0
    for k, (u, half, nodes) in enumerate(steps):
        first = (eye + half) @ pre[k] if half is not None else u @ pre[k]
        err += unit * (_norm(first[nodes]) + _norm(pre[k + 1][nodes])) * _norm(post[k][:, nodes])
    return pre[-1], err


@pytest.mark.parametrize("P,L,which", [(64, 4, 0), (32, 3, 1)])
def test_bounds_cover_the_rounding(P, L, which):
    text = open(SRC).read()
    ERR, ROUND = [[float(x) for x in re.search(name + r" = P == 64 \? (\S+) : ([^;,]+)[;,]", text).groups()][which]
                  for name in ("ERR", "ROUND")]
    inv, e32 = _line(P, L, True, 2.0 ** -24)
    x = np.random.default_rng(0).normal(size=P + 1)
    assert np.allclose(O.dwt(np.outer(x, x), "bl53", P, L, inverse=True), np.outer(inv @ x, inv @ x))
    gain = np.linalg.svd(inv, compute_uv=False)
    N, low = gain[0], gain[-1]
    # two passes, the other axis's norm beside each; the coefficients' own rounding
    assert 2 * e32 * N + 2.0 ** -24 * N * N <= ERR
    fwd, e64f = _line(P, L, False, 2.0 ** -53)
    _, e64i = _line(P, L, True, 2.0 ** -53)
    assert 2 * e64i * N / low ** 2 + 2 * e64f * _norm(fwd) * N * N <= ROUND


@pytest.mark.parametrize("P,L,ERR", [(64, 4, 2.7e-5), (32, 3, 1.1e-5)])
def test_fp32_transform_stays_below_the_bound(P, L, ERR):
    rng = np.random.default_rng(P)
    worst = 0.0
    for kind in range(12):
        c = rng.normal(size=(P + 1, P + 1)) * 10.0 ** rng.uniform(-3 * (kind % 4), 0, size=(P + 1, P + 1))
        if kind >= 8:
            c = np.abs(c)
        c[:: 1 << L, :: 1 << L] = 0.0
        exact = O.dwt(c, "bl53", P, L, inverse=True)
        t = c.astype(np.float32)
        for _ in range(2):  # columns, then rows
            for u, half, nodes in _steps(P, L, True):
                if half is not None:
                    t[nodes] = np.float32(t[nodes] + (half @ t)[nodes])
                    t[nodes] = np.float32(t[nodes] + ((u - half) @ t)[nodes])
                else:
                    t[nodes] = np.float32(t[nodes] + np.float32((u @ t)[nodes]))
            t = np.ascontiguousarray(t.T)
        worst = max(worst, np.linalg.norm(t - exact) / np.linalg.norm(c))
    assert 0.0 < worst < ERR / 20
