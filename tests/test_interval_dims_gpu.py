"""Every draw from fhat(.|x), at each number of coordinates the sampling kernels are
built for and for both kernels, against FP64 cumulative weights.  A target closer to a
boundary than SLACK of the total may fall on either side of it: 2^-19, for FP32 weights
(distances of up to 40 dimensions 2^-20 of the few powers of two they are worth) and
running sums of 32-point segments.  All other draws are the one value."""
from statistics import NormalDist

import numpy as np
import pytest

from paper_1206_5278_gb300 import cde
from test_interval_gpu import _uniforms

pytestmark = pytest.mark.gpu

SLACK = 2.0 ** -19


@pytest.fixture(scope="module")
def ctx():
    c = cde.cde_init(0)
    yield c
    cde.cde_shutdown(c)


def _take(left, v):
    """Remove the entry of the sorted list nearest v; False where none is within 1e-5."""
    k = int(np.searchsorted(left, v))
    best = min((j for j in (k - 1, k) if 0 <= j < len(left)), key=lambda j: abs(left[j] - v), default=None)
    if best is None or abs(left[best] - v) > 1e-5:
        return False
    del left[best]
    return True


@pytest.mark.parametrize("kernel", ["gauss", "epan"])
@pytest.mark.parametrize("d", [3, 7, 12, 20, 40])
@pytest.mark.parametrize("N,Q,S", [(300, 1, 1), (1000, 3, 5), (2049, 130, 200)])
def test_each_draw(ctx, kernel, d, N, Q, S):
    rng = np.random.default_rng(1000 * d + N)
    x = (rng.standard_normal((N, d)) / np.sqrt(d)).astype(np.float32)
    xq = (rng.standard_normal((Q, d)) / np.sqrt(d)).astype(np.float32)
    y = rng.uniform(-3.0, 3.0, N).astype(np.float32)
    h1, h2, seed = (0.7, 0.01, 5) if kernel == "gauss" else (1.5, 0.01, 5)
    ds = cde.cde_create_dataset(ctx, x, y, kernel=kernel)
    _, _, got = cde.cde_cond_interval(ctx, ds, h1, h2, xq, S=S, alpha=0.1, seed=seed, samples=True)
    cde.cde_destroy_dataset(ctx, ds)
    either = 0
    for q in sorted({0, Q // 2, Q - 1}):
        d2 = ((x.astype(np.float64) - xq[q].astype(np.float64)) ** 2).sum(1)
        w = np.exp(-(d2 - d2.min()) / (2 * h1 * h1)) if kernel == "gauss" else np.maximum(1.0 - d2 / (h1 * h1), 0.0)
        c = np.cumsum(w)
        live = np.nonzero(w > 0)[0]
        k0 = 2 * (np.uint64(q) * np.uint64(S) + np.arange(S, dtype=np.uint64))
        t = np.sort(_uniforms(seed, k0)).astype(np.float64) * c[-1]
        V = _uniforms(seed, k0 + np.uint64(1)).astype(np.float64)
        off = np.array([NormalDist().inv_cdf(v) for v in V]) if kernel == "gauss" else 2 * np.sin(np.arcsin(2 * V - 1) / 3)
        first = np.searchsorted(c, t - SLACK * c[-1], side="right")
        last = np.searchsorted(c, t + SLACK * c[-1], side="right")
        left = sorted(got[q].astype(np.float64).tolist())
        for s in np.argsort(last - first, kind="stable"):   # the certain ones first
            cand = live[(live >= first[s]) & (live <= last[s])]
            either += cand.size > 1
            assert any(_take(left, y[i] + h2 * off[s]) for i in (cand if cand.size else live[-1:])), (q, s)
        assert not left
    assert either <= max(1, S // 10)      # the check decides nearly every draw
