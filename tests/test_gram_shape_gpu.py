"""d >= 16 grids (the Gram-form tile kernel) over the grid shapes and the numbers of
rows at which the block shape changes: every row's terms against the FP64 oracle,
and the scores against the sum of the rows."""
import numpy as np
import pytest

from oracle import oracle
from oracle.fp32_bounds import rows_within_bound
from paper_1206_5278_gb300 import cde, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = cde.cde_init(0)
    yield c
    cde.cde_shutdown(c)


# one unit short of and past a full wave of the narrow shapes' units (128 and 64 rows x
# 152), a few rows, and the wide grids; lo = 0.05 leaves most cells to the recomputation
@pytest.mark.parametrize("lo", [0.05, 0.8])
@pytest.mark.parametrize("N,d,G1,G2", [(67, 16, 1, 1), (1021, 17, 8, 8), (2433, 16, 5, 7), (4999, 24, 8, 3),
                                       (9729, 16, 8, 8), (19457, 16, 4, 8), (3001, 33, 16, 8), (2600, 20, 9, 12),
                                       (1500, 16, 17, 5), (1201, 19, 31, 32)])
def test_gram_rows_over_shapes(ctx, N, d, G1, G2, lo):
    x, y = synth.gmm_sine(N, d, seed=N + d)
    h1, h2 = np.geomspace(lo, 3.0, G1), np.geomspace(lo / 4, 1.0, G2)
    x64 = (x.astype(np.float64) - x.astype(np.float64).mean(0)) / x.astype(np.float64).std(0, ddof=1)
    ds = cde.cde_create_dataset(ctx, x, y, standardize=True)
    rows = np.unique(np.linspace(0, N - 1, 40).astype(np.int64))
    got = cde.cde_loo_rows(ctx, ds, h1, h2, rows)
    ref = oracle.loo_rows(x, y, h1, h2, rows=rows, standardize_x=True)[0]
    ok, worst = rows_within_bound(got, ref, x64, y, h1, h2, rows, gram=True)
    assert ok, worst
    Lc, _ = cde.cde_loo_loglik(ctx, ds, h1, h2)
    ell = cde.cde_loo_rows(ctx, ds, h1, h2, np.arange(N))
    tot, tot_abs = ell.sum(0), np.abs(ell).sum(0)
    assert np.isfinite(tot).all()
    # FP64 summation order, and recomputed cells (terms under 2^-32 of a sum, the last bit
    # of its FP32 logarithm) that meet other rows in their unit
    assert np.all(np.abs(Lc - tot) <= 1e-12 * tot_abs + 1e-6 * N)
    cde.cde_destroy_dataset(ctx, ds)
