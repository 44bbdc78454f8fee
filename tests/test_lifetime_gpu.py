"""A dataset destroyed, or a whole context shut down, right after calls with device
outputs on a caller's stream: the calls finish on the dataset's memory first."""
import numpy as np
import pytest

from paper_1206_5278_gb300 import cde, synth

pytestmark = pytest.mark.gpu


class _Calls:
    """Calls of each kind with device outputs (about 30 ms of kernels), and what they use."""

    def __init__(self, x):
        import torch
        self.h1, self.h2 = synth.bandwidth_grid(0.05, 2.0, 32), synth.bandwidth_grid(0.01, 1.0, 32)
        self.xq, self.yg = torch.from_numpy(x[:64].copy()).cuda(), torch.linspace(-2, 2, 33, device="cuda")
        self.out = [torch.zeros(32 * 32, dtype=torch.float64, device="cuda"),
                    torch.zeros(3, dtype=torch.float64, device="cuda"), torch.zeros((64, 33), device="cuda")]
        self.stream = torch.cuda.Stream()
        torch.cuda.synchronize()

    def enqueue(self, ctx, ds):
        for _ in range(2):
            cde.cde_loo_loglik(ctx, ds, self.h1, self.h2, L_cond_out=self.out[0], stream=self.stream)
        cde.cde_loo_grad(ctx, ds, 0.3, 0.1, out3=self.out[1], stream=self.stream)
        cde.cde_density(ctx, ds, 0.3, 0.1, self.xq, self.yg, f_out=self.out[2], stream=self.stream)

    def result(self):
        self.stream.synchronize()
        r = [t.cpu().numpy().copy() for t in self.out]
        for t in self.out:
            t.zero_()
        return r


@pytest.mark.parametrize("how", ["shutdown", "destroy"])
def test_calls_in_flight_finish_first(how):
    import torch
    x, y = synth.gmm_sine(20011, 5, seed=3)
    other = synth.gmm_sine(20011, 5, seed=4)
    ctx = cde.cde_init(0)
    ds = cde.cde_create_dataset(ctx, x, y, standardize=True)
    calls = _Calls(x)
    calls.enqueue(ctx, ds)
    want = calls.result()
    torch.cuda.synchronize()
    calls.enqueue(ctx, ds)
    if how == "shutdown":
        cde.cde_shutdown(ctx)
        ctx = cde.cde_init(0)
    else:
        cde.cde_destroy_dataset(ctx, ds)
    for _ in range(3):   # whatever takes the memory next
        cde.cde_create_dataset(ctx, *other, standardize=True)
    for a, b in zip(calls.result(), want):
        assert np.array_equal(a, b)
    cde.cde_shutdown(ctx)
