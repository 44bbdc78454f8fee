"""Recomputed cells of the d >= 16 kernel on rows in descending order of their exponent
(every point could become the recomputation's new anchor): 2,000 additions rounded
independently are off by sqrt(2000) 2^-24 = 2.7e-6; with the terms' own error (2^-22 for
the exponentials, 2^-19 as the direct kernels' cells) 5e-6.  On tied points, where every
addition would round the same way, within the direct kernels' 2^-19."""
import pytest

from test_recompute_sums_gpu import _error, ctx  # noqa: F401  (ctx: the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G1,G2,d", [(16, 8, 20), (16, 16, 16), (32, 32, 33)])
def test_sorted_rows(ctx, G1, G2, d):  # noqa: F811
    assert _error(ctx, "sorted", 20000, G1, G2, d) <= 5e-6


@pytest.mark.parametrize("G1,G2,d", [(16, 8, 20), (16, 16, 16), (32, 32, 33)])
def test_tied_points(ctx, G1, G2, d):  # noqa: F811
    assert _error(ctx, "tied", 20000, G1, G2, d) <= 2.0 ** -19
