"""The d_x > 8 nearest-distance kernels at the edges of their tiles (128 rows,
64 points, splits of several tiles): dataset shifts and query shifts."""
import numpy as np
import pytest

from oracle import oracle
from paper_1206_5278_gb300 import cde, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = cde.cde_init(0)
    yield c
    cde.cde_shutdown(c)


@pytest.mark.parametrize("N,d", [(2, 9), (63, 64), (64, 10), (65, 33), (127, 16), (129, 9), (1025, 11), (2500, 17)])
def test_nearest_neighbours(ctx, N, d):
    """FP32 differences, squares and running sums with one rounding per dimension
    (emulated in FP64, which may round a sum twice: at most one ulp per dimension)."""
    x, y = synth.random_small(N, d, seed=N + d)
    y = np.round(y, 1)      # ties in y: the smallest x distance of the tied points
    ds = cde.cde_create_dataset(ctx, x, y)
    acc = np.zeros((N, N), np.float32)
    for c in range(d):
        q = (x[:, None, c] - x[None, :, c]).astype(np.float32)
        acc = (q.astype(np.float64) ** 2 + acc).astype(np.float32)
    np.fill_diagonal(acc, np.inf)
    dy2 = ((y[:, None] - y[None, :]).astype(np.float32) ** 2).astype(np.float32)
    np.fill_diagonal(dy2, np.inf)
    mx, my = cde.cde_dataset_nn(ctx, ds)
    qx, qy = cde.cde_dataset_nn_other(ctx, ds)
    np.testing.assert_allclose(mx, acc.min(1), rtol=d * 2.0 ** -23, atol=0)
    np.testing.assert_array_equal(my, dy2.min(1))
    np.testing.assert_allclose(qx, np.where(dy2 == my[:, None], acc, np.inf).min(1), rtol=d * 2.0 ** -23, atol=0)
    assert np.mean(qy == np.where(acc == acc.min(1, keepdims=True), dy2, np.inf).min(1)) >= 0.99
    cde.cde_destroy_dataset(ctx, ds)


@pytest.mark.parametrize("Q,N,d", [(1, 65, 9), (129, 64, 12), (257, 1000, 40)])
def test_query_shift_pins_the_density(ctx, Q, N, d):
    """At a bandwidth far below the point spacing a wrong shift over- or underflows
    every x factor."""
    x, y = synth.gmm_sine(N, d, seed=N + d)
    xq = synth.query_points(x, Q, seed=d)
    yg = synth.y_grid(y, 0.3, 33)
    ds = cde.cde_create_dataset(ctx, x, y, standardize=True)
    f = cde.cde_density(ctx, ds, 0.1, 0.3, xq, yg)
    ref = oracle.density(x, y, 0.1, 0.3, xq, yg, standardize_x=True)
    assert np.all(np.abs(f - ref) <= 1e-4 * ref.max(1, keepdims=True))
    cde.cde_destroy_dataset(ctx, ds)
