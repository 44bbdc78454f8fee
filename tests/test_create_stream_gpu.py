"""A dataset made from CUDA tensors that torch's current stream is still writing."""
import numpy as np
import pytest

from paper_1206_5278_gb300 import cde, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [False, True])
@pytest.mark.parametrize("strided", [False, True])
def test_arrays_in_the_making(side, strided):
    import torch
    ctx = cde.cde_init(0)
    x, y = synth.gmm_sine(3001, 3, seed=8)
    want = cde.cde_dataset_nn(ctx, cde.cde_create_dataset(ctx, x, y, standardize=True))
    hx, hy = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    dx = torch.rand((3, 3001) if strided else (3001, 3), device="cuda")
    dy = torch.rand(3001, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.default_stream()):
        torch.cuda._sleep(100_000_000)          # about 50 ms
        tx = dx.t() if strided else dx
        tx.copy_(hx)
        dy.copy_(hy)
        ds = cde.cde_create_dataset(ctx, tx, dy, standardize=True)
    for a, b in zip(cde.cde_dataset_nn(ctx, ds), want):
        assert np.array_equal(a, b)
    cde.cde_shutdown(ctx)
