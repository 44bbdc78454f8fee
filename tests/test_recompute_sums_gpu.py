"""Precision of the sums of recomputed cells (cells whose shifted numerator underflows):
a left-out row far from everything, thousands of points that carry its cells, either
tied (every addition would round the same way) or in descending order of their exponent
(every point would become the recomputation's new anchor).

Distances and coefficients are exact here: coordinates on a coarse binary grid or the
FP32 squares of the differences, log2(e)/(2 h^2) a short binary fraction.  What is left
of a direct cell's error: the terms' exponentials 2^-22, 32 FP32 additions 2^-20, the
logarithms and the denominator (one point carries it) 2^-21, the sums put together
2^-22: 2^-19 in all."""
import numpy as np
import pytest

from paper_1206_5278_gb300 import cde

pytestmark = pytest.mark.gpu

L2E = 1.4426950408889634


@pytest.fixture(scope="module")
def ctx():
    c = cde.cde_init(0)
    yield c
    cde.cde_shutdown(c)


def _rows(kind, n):
    """Points beside the left-out one at (0, 0): its x-nearest (0, 16) and y-nearest
    (16, 0), and n that carry its cells."""
    x, y = np.full(n, 8.0, np.float32), np.full(n, 8.0, np.float32)
    if kind == "tied":     # one point a chunk at the minimum, in every warp's first chunk; the rest tied behind it
        x[:] = 8.125
        x[np.arange(8) * 64] = 8.0
    else:
        y = np.linspace(9.0, 8.0, n).astype(np.float32)
    return np.concatenate([x, [0.0, 16.0, 0.0]]).astype(np.float32), np.concatenate([y, [16.0, 0.0, 0.0]]).astype(np.float32)


def _error(ctx, kind, n, G1, G2, d):
    x, y = _rows(kind, n)
    A, B = (96.0 + 3.0 * np.arange(G1)) / 128.0, (100.0 + 5.0 * (np.arange(G2) % 16)) / 128.0
    h1, h2 = np.sqrt(L2E / (2.0 * A)), np.sqrt(L2E / (2.0 * B))
    xd = np.zeros((x.size, d), np.float32)
    xd[:, 0] = x
    ds = cde.cde_create_dataset(ctx, xd, y, standardize=False)
    got = cde.cde_loo_rows(ctx, ds, h1, h2, [x.size - 1])[0]
    cde.cde_destroy_dataset(ctx, ds)
    X, Y = (x[:-1] * x[:-1]).astype(np.float64), (y[:-1] * y[:-1]).astype(np.float64)
    ex = -A[:, None] * X
    lnB = np.log(np.exp2(ex).sum(1))
    worst = 0.0
    for l in range(min(G2, 16)):
        e = ex - B[l] * Y
        top = e.max(1, keepdims=True)
        ref = np.log(np.exp2(e - top).sum(1)) + top[:, 0] * np.log(2.0) - lnB - np.log(np.sqrt(2.0 * np.pi) * h2[l])
        worst = max(worst, np.abs(got[:, l::16] - ref[:, None]).max())
    return worst


@pytest.mark.parametrize("kind,n", [("tied", 20000), ("sorted", 100000)])
@pytest.mark.parametrize("G1,G2,d", [(4, 4, 1), (8, 8, 12), (16, 8, 3), (16, 16, 2), (32, 16, 1), (32, 32, 2)])
def test_sums_of_recomputed_cells(ctx, kind, n, G1, G2, d):
    assert _error(ctx, kind, n, G1, G2, d) <= 2.0 ** -19
