"""The checked build (device index checks) on the kernels of more dimensions: the d >= 16
grid over its block shapes with recomputed cells, the shift tiles of d > 8 datasets and
queries, the sampling kernels, gradients with few and with most rows recomputed.  No
check fails, and the results are the normal library's."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import json, sys
import numpy as np
sys.path.insert(0, ROOT_PATH)
from paper_1206_5278_gb300 import cde, synth

def L(a):
    return np.asarray(a, dtype=np.float64).ravel().tolist()

ctx = cde.cde_init(0)
out = {}
for n, d, g1, g2, k in [(2, 16, 8, 8, "gauss"), (129, 17, 5, 7, "gauss"), (1031, 20, 8, 8, "gauss"), (777, 33, 16, 16, "gauss"),
                        (515, 64, 32, 32, "gauss"), (640, 24, 33, 9, "gauss"), (300, 20, 16, 32, "epan")]:
    x, y = synth.random_small(n, d, seed=n + d)
    ds = cde.cde_create_dataset(ctx, x, y, standardize=True, kernel=k)
    wide = 6.0 if k == "epan" else 1.0
    h1, h2 = wide * synth.bandwidth_grid(0.2, 3.0, g1), wide * synth.bandwidth_grid(0.01, 2.0, g2)
    Lc, Le = cde.cde_loo_loglik(ctx, ds, h1, h2)
    out["loo_%d_%d" % (n, d)] = L(Lc) + L(Le)
    out["rows_%d_%d" % (n, d)] = L(cde.cde_loo_rows(ctx, ds, h1, h2, [0, n // 2, n - 1]))
    cde.cde_destroy_dataset(ctx, ds)
for d in (9, 12, 20, 40, 64):
    for k in ("gauss", "epan"):
        x, y = synth.random_small(901, d, seed=d)
        ds = cde.cde_create_dataset(ctx, x, y, standardize=True, kernel=k)
        h1 = 1.0 if k == "gauss" else 8.0
        xq = synth.query_points(x, 131, seed=1)
        out["density_%d_%s" % (d, k)] = L(cde.cde_density(ctx, ds, h1, 0.2, xq, synth.y_grid(y, 0.2, 70)))
        m, f = cde.cde_cond_stats(ctx, ds, h1, 0.2, xq, y[:131])
        out["stats_%d_%s" % (d, k)] = L(m) + L(f)
        lo, hi, sm = cde.cde_cond_interval(ctx, ds, h1, 0.2, xq, S=150, alpha=0.1, seed=3, samples=True)
        out["interval_%d_%s" % (d, k)] = L(lo) + L(hi) + L(sm)
        cde.cde_destroy_dataset(ctx, ds)
for n, d, h1, h2 in [(2, 3, 0.02, 0.002), (63, 5, 0.02, 0.002), (2503, 3, 0.02, 0.002), (2503, 3, 0.3, 0.05),
                     (9300, 4, 0.1, 0.01), (1025, 12, 0.1, 0.01), (3001, 33, 0.3, 0.005)]:
    x, y = synth.gmm_sine(n, d, seed=n)
    ds = cde.cde_create_dataset(ctx, x, y, standardize=n > 2)
    out["grad_%d_%d_%g" % (n, d, h1)] = L(cde.cde_loo_grad_rows(ctx, ds, h1, h2)) + L(cde.cde_loo_grad(ctx, ds, h1, h2))
    cde.cde_destroy_dataset(ctx, ds)
code, enabled = cde.cde_check_status(ctx)
out["check"] = [code, enabled]
cde.cde_shutdown(ctx)
print(json.dumps(out))
'''.replace("ROOT_PATH", repr(ROOT))


def _run(variant):
    env = dict(os.environ)
    env.pop("CDE_LIBRARY", None)
    if variant == "checked":
        env["CDE_LIBRARY"] = "checked"
    r = subprocess.run([sys.executable, "-c", SCRIPT], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_no_failed_check_and_the_same_results():
    from paper_1206_5278_gb300 import _build
    _build.build(checks=True)
    normal, checked = _run("normal"), _run("checked")
    assert normal["check"] == [0, False]
    assert checked["check"] == [0, True], "failed device index check, code %d" % checked["check"][0]
    assert normal.keys() == checked.keys()
    for key in normal.keys() - {"check"}:
        assert [repr(v) for v in normal[key]] == [repr(v) for v in checked[key]], key
