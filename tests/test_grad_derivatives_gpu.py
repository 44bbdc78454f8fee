"""Per-row derivatives of the gradient: no row, some rows and most rows recomputed (in
groups of four over one or several point ranges), on the direct and the tensor-core
kernel.  Coordinates on a coarse binary grid and log2(e)/(2 h^2) whole, so distances and
coefficients are exact (also as TF32 products); what is left of a sum's relative error:
exponent arguments up to 2^7, rounded, 2^-17, and at most 256 FP32 additions in a row
2^-16: EPS = 2^-15 with room for the merges."""
import numpy as np
import pytest

from oracle import oracle
from paper_1206_5278_gb300 import cde

pytestmark = pytest.mark.gpu

L2E, EPS = 1.4426950408889634, 2.0 ** -15


@pytest.fixture(scope="module")
def ctx():
    c = cde.cde_init(0)
    yield c
    cde.cde_shutdown(c)


@pytest.mark.parametrize("A,B", [(1, 2), (24, 512), (64, 1024), (128, 4096)])
@pytest.mark.parametrize("N,d", [(129, 1), (257, 12), (1025, 3), (2503, 3), (4100, 5), (3001, 20)])
def test_derivative_columns(ctx, N, d, A, B):
    rng = np.random.default_rng(N + d)
    x, y = (rng.integers(-16, 17, (N, d)) / 8).astype(np.float32), (rng.integers(-64, 65, N) / 32).astype(np.float32)
    h1, h2 = np.sqrt(L2E / (2 * A)), np.sqrt(L2E / (2 * B))
    ds = cde.cde_create_dataset(ctx, x, y)
    got = cde.cde_loo_grad_rows(ctx, ds, h1, h2)
    rows = np.arange(0, N, max(1, N // 300))
    _, ref = oracle.grad(x, y, h1, h2, rows=rows, per_row=True)
    X = ((x[rows, None].astype(np.float64) - x[None]) ** 2).sum(2)
    Y = (y[rows, None].astype(np.float64) - y[None]) ** 2
    own = np.arange(rows.size), rows
    eB = -A * X
    eB[own] = -np.inf
    e = eB - B * Y
    v, u = np.exp2(e - e.max(1, keepdims=True)), np.exp2(eB - eB.max(1, keepdims=True))
    mean = lambda w, t: (w * t).sum(1) / w.sum(1)   # noqa: E731
    tol = np.stack([2 * EPS * np.ones(rows.size), 2 * EPS * (mean(v, X) + mean(u, X)) / h1 ** 2,
                    2 * EPS * mean(v, Y) / h2 ** 2], 1) + 1e-12 * np.abs(ref)
    assert np.all(np.abs(got[rows] - ref) <= tol), (np.abs(got[rows] - ref) / tol).max(0)
    cde.cde_destroy_dataset(ctx, ds)
