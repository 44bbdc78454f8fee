"""Grids of at most 8 x 8 bandwidths (the packed tile body): every row's terms
are bitwise those of the same bandwidths inside a wider grid, which runs on the
16-row tile body, and the scores match the FP64 oracle."""
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


# chunk (64 points), unit (8 rows) and warp-range edges; every packed shape, full and
# ragged; the register (d <= 8) and the loaded (d > 8) coordinates
@pytest.mark.parametrize("kernel", ["gauss", "epan"])
@pytest.mark.parametrize("N,d,G1,G2", [(2, 1, 1, 1), (9, 2, 4, 4), (63, 1, 4, 5), (65, 8, 8, 8), (513, 9, 3, 2),
                                       (700, 13, 8, 4), (1203, 5, 7, 8), (2000, 1, 8, 8), (520, 15, 5, 3)])
def test_packed_rows_equal_the_wide_grid(ctx, kernel, N, d, G1, G2):
    x, y = synth.random_small(N, d, seed=N + d)
    h1, h2 = synth.bandwidth_grid(0.3, 3.0, 9), synth.bandwidth_grid(0.1, 2.0, 8)
    if kernel == "epan":
        h1, h2 = 4.0 * h1, 4.0 * h2
    ds = cde.cde_create_dataset(ctx, x, y, standardize=False, kernel=kernel)
    rows = np.arange(N)
    wide = cde.cde_loo_rows(ctx, ds, h1, h2, rows)[:, :G1, :G2]          # 9 x 8: the 16-row body
    h1, h2 = h1[:G1], h2[:G2]
    got = cde.cde_loo_rows(ctx, ds, h1, h2, rows)
    same = got == wide
    if kernel == "epan":
        assert same.all()
    else:
        # recomputed cells may see other candidate points: terms under 2^-32 of the sum
        # and the last bit of its FP32 logarithm
        with np.errstate(invalid="ignore"):
            assert np.all(same | (np.abs(got - wide) <= 1e-6)) and same.mean() > 0.5
        ref = oracle.loo_rows(x, y, h1, h2, rows=rows)[0]
        ok, worst = rows_within_bound(got, ref, x.astype(np.float64), y, h1, h2, rows)
        assert ok, worst
    Lc, _ = cde.cde_loo_loglik(ctx, ds, h1, h2)
    tot = got.sum(0)
    fin = np.isfinite(tot)
    assert np.array_equal(np.isfinite(Lc), fin)
    assert np.all(np.abs(Lc[fin] - tot[fin]) <= 1e-12 * np.abs(got).sum(0)[fin])   # FP64 summation order only
    cde.cde_destroy_dataset(ctx, ds)


@pytest.mark.parametrize("G1,G2,d", [(4, 4, 12), (8, 8, 3), (16, 8, 9), (16, 16, 5), (32, 8, 2), (16, 32, 4), (32, 16, 12)])
def test_one_pass_recomputation(ctx, G1, G2, d):
    """Bandwidths so small that most cells of most rows underflow (units with more
    recomputed cells than one round holds at 16 x 8), on sizes off the chunk grid."""
    N = 713
    x, y = synth.gmm_sine(N, d, seed=40 + d)
    h1, h2 = synth.bandwidth_grid(0.03, 0.3, G1), synth.bandwidth_grid(0.003, 0.05, G2)
    x64 = (x.astype(np.float64) - x.astype(np.float64).mean(0)) / x.astype(np.float64).std(0, ddof=1)
    ds = cde.cde_create_dataset(ctx, x, y, standardize=True)
    rows = np.arange(0, N, 3)
    got = cde.cde_loo_rows(ctx, ds, h1, h2, rows)
    ref = oracle.loo_rows(x, y, h1, h2, rows=rows, standardize_x=True)[0]
    ok, worst = rows_within_bound(got, ref, x64, y, h1, h2, rows)
    assert ok, worst
    cde.cde_destroy_dataset(ctx, ds)
