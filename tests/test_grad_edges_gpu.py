"""Gradient at the edges of its launches: point splits down to one tile and two
rows per thread (small N), rows recomputed in groups of four over several point
ranges, the block sums of the rows."""
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


# (0.02, 0.002): most rows are listed for the joint-shift recomputation; (0.5, 0.2): none
@pytest.mark.parametrize("h1,h2", [(0.02, 0.002), (0.5, 0.2)])
@pytest.mark.parametrize("N,d", [(2, 1), (5, 4), (129, 8), (257, 12), (1025, 3), (2503, 3), (4100, 5)])
def test_gradient_rows(ctx, N, d, h1, h2):
    x, y = synth.gmm_sine(N, d, seed=N + d)
    ds = cde.cde_create_dataset(ctx, x, y, standardize=True)
    got = cde.cde_loo_grad_rows(ctx, ds, h1, h2)
    rows = np.arange(0, N, max(1, N // 300))
    _, ref = oracle.grad(x, y, h1, h2, rows=rows, standardize_x=True, per_row=True)
    # FP32 squared distances are off by a few 2^-24 of |x|^2 + d^2: in the log-weights of
    # Eq. 1 by that over 2 h1^2 (2 h2^2 for y); a row term is a difference of two such means
    z = oracle.standardize(x)
    reach = (np.abs(z).max(1) ** 2 * d * 8 + 4)[rows] * 2.0 ** -22
    tol = 2e-5 * (1 + np.abs(ref[:, 0])) + reach / (2 * h1 * h1) + np.abs(y).max() ** 2 * 2.0 ** -21 / (2 * h2 * h2)
    assert np.all(np.abs(got[rows, 0] - ref[:, 0]) <= tol)
    out = cde.cde_loo_grad(ctx, ds, h1, h2)
    np.testing.assert_allclose(out, got.sum(0), rtol=0, atol=1e-12 * np.abs(got).sum(0).max())
    assert np.array_equal(cde.cde_loo_grad_rows(ctx, ds, h1, h2), got)      # whatever order the list was written in
    cde.cde_destroy_dataset(ctx, ds)
