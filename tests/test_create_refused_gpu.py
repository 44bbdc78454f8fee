"""A dataset that is refused (a non-finite value in device arrays, a dimension
without spread) is refused before the O(N^2 d) work, with the same errors."""
import time

import numpy as np
import pytest

from paper_1206_5278_gb300 import cde

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = cde.cde_init(0)
    yield c
    cde.cde_shutdown(c)


def _seconds(ctx, x, y, text):
    best = np.inf
    for _ in range(4):
        t = time.perf_counter()
        if text:
            with pytest.raises(cde.CdeError, match=text) as e:
                cde.cde_create_dataset(ctx, x, y, standardize=True)
            assert e.value.status == cde.CDE_EINVAL
        else:
            cde.cde_destroy_dataset(ctx, cde.cde_create_dataset(ctx, x, y, standardize=True))
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("N,d", [(160001, 5), (100003, 32)])   # the kernels of d <= 8 and d > 8
def test_refused_without_the_shifts(ctx, N, d):
    import torch
    g = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn((N, d), generator=g, device="cuda")
    y = torch.randn(N, generator=g, device="cuda")
    whole = _seconds(ctx, x, y, None)
    nan, flat, yinf = x.clone(), x.clone(), y.clone()
    nan[N // 2, d - 1] = float("nan")
    flat[:, d // 2] = 1.5
    yinf[N - 1] = float("inf")
    both = nan.clone()
    both[:, 0] = 0.25
    torch.cuda.synchronize()
    for bad in ((nan, y, "non-finite"), (x, yinf, "non-finite"), (flat, y, "zero spread"), (both, y, "non-finite")):
        assert _seconds(ctx, *bad) <= 0.5 * whole
    # without standardising, a dimension without spread is no error
    cde.cde_destroy_dataset(ctx, cde.cde_create_dataset(ctx, flat, y, standardize=False))
