"""Memory booked for a selection job covers what its gradient steps allocate."""
import numpy as np
import pytest

from paper_1206_5278_gb300 import cde, synth
from paper_1206_5278_gb300.serve import Server

pytestmark = pytest.mark.gpu


def _booked(ctx, ds, hi):
    """The smallest budget that admits the job: a bisection over the server's answers."""
    h = synth.bandwidth_grid(0.1, 1.0, 4)
    lo = 0
    while hi - lo > 1024:
        mid = (lo + hi) // 2
        srv = Server(ctx, n_streams=1, job_mem_budget=mid)
        try:
            st, t = srv.try_submit(Server.select_request(ds, h, h, 0))
            if st == cde.CDE_OK:
                t.wait()
        finally:
            srv.stop()
        assert st in (cde.CDE_OK, cde.CDE_ENOMEM)
        if st == cde.CDE_OK:
            hi = mid
        else:
            lo = mid
    return hi


@pytest.mark.parametrize("N,d", [(2, 1), (40, 3), (9216, 3), (9216, 64)])
def test_selection_books_its_gradient(N, d):
    import torch
    ctx = cde.cde_init(0)
    x, y = synth.random_small(N, d, seed=N)
    ds = cde.cde_create_dataset(ctx, x, y)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # partial sums: six floats per row and point split, or per recomputed row and range
    # (four CTAs per SM, four rows each, two items a CTA); three doubles per row; at
    # d >= 16 the points' split coordinates, two words each, padded to 16, 32 or 64
    need = 24 * (N + 4 + 32 * sms) + 24 * N
    if d >= 16:
        need += 8 * 64 * ((N + 255) // 256 * 256)
    assert _booked(ctx, ds, 1 << 28) >= need
    cde.cde_destroy_dataset(ctx, ds)
    cde.cde_shutdown(ctx)
