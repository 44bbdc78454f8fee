"""Scratch freed by a call stays mapped for the next one however large the resident
datasets are, and the memory of destroyed datasets goes back to the device."""
import numpy as np
import pytest

from paper_1206_5278_gb300 import cde

pytestmark = pytest.mark.gpu


def test_scratch_is_kept_beside_large_datasets():
    import torch
    ctx = cde.cde_init(0)
    # (an Epanechnikov dataset has no shifts: 430 MB resident at once, from device arrays)
    x, y = torch.rand((2000003, 48), device="cuda"), torch.rand(2000003, device="cuda")
    torch.cuda.synchronize()
    large = cde.cde_create_dataset(ctx, x, y, kernel="epan")
    small = cde.cde_create_dataset(ctx, np.random.rand(3000, 2).astype(np.float32), np.random.rand(3000).astype(np.float32))
    xq, yg = np.random.rand(60000, 2).astype(np.float32), np.linspace(0.0, 1.0, 256).astype(np.float32)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0] >> 20

    start = free()
    cde.cde_density(ctx, small, 0.3, 0.1, xq, yg)          # 61 MB of output and some of partial sums
    kept = free()
    assert 40 <= start - kept <= 256
    cde.cde_density(ctx, small, 0.3, 0.1, xq, yg)
    assert free() == kept
    cde.cde_destroy_dataset(ctx, large)
    cde.cde_density(ctx, small, 0.3, 0.1, xq[:5], yg)
    assert free() - kept >= 200
    cde.cde_destroy_dataset(ctx, small)
    cde.cde_shutdown(ctx)
