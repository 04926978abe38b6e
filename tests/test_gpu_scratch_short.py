"""Scratch that a call can do without (GPU): the 16-bit forms list their moved rows
(24 bytes a row) where there is room.  What fits without the list still runs,
with the same results, and a server still admits it."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1108_1351_gb300 as km  # noqa: E402
from paper_1108_1351_gb300 import synth  # noqa: E402

CASE = r"""
import os, sys, torch
sys.path.insert(0, ROOT)
import paper_1108_1351_gb300 as km
from paper_1108_1351_gb300 import synth
assert km.LIB_PATH.endswith("libkmeans2_debug.so")
n, d, k = 400_000, 64, 600
X = synth.vmf_mixture(n, d, k, 3, device="cuda")
C = X[:k].double().contiguous()
calls = {"step": lambda: km.step(X, C, precision="bf16")}
for p in ("bf16", "fp16", "auto"):
    calls[p] = lambda p=p: km.fit(X, k, 0.02, 1, 1e-6, 6, precision=p)
def least(f):
    lo, hi = 0, 1 << 30                    # refused at lo, runs at hi
    while hi - lo > 1 << 17:
        mid = (lo + hi) // 2
        os.environ["KMEANS2_DEBUG_SCRATCH_BYTES"] = str(mid)
        try:
            f()
            hi = mid
        except km.KMeans2Error as e:
            assert e.status == -2, e
            lo = mid
    os.environ["KMEANS2_DEBUG_SCRATCH_BYTES"] = str(hi)
    r = f()
    del os.environ["KMEANS2_DEBUG_SCRATCH_BYTES"]
    return hi, r
for name, f in calls.items():
    want = f()
    need, got = least(f)
    if name == "step":
        assert torch.equal(got[1], want[1]) and torch.equal(got[0], want[0]) and got[2:] == want[2:]
        # the tiles, ||x||^2, the recheck list, the centers' copies; not 24 bytes a row more
        assert need <= n * (4 * d + 4 + 4) + 24 * k * d * 4 + (2 << 20), need
    else:
        assert torch.equal(got.labels, want.labels) and torch.equal(got.centers, want.centers) and got.J == want.J
        assert need <= km.footprint(n, d, k, 0.02, 6, precision=name) - 24 * n, (name, need)
print("ok")
"""


def test_calls_run_without_room_for_the_list():
    from paper_1108_1351_gb300 import build
    build.build(debug=True)
    env = dict(os.environ, KMEANS2_DEBUG="1")
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + CASE], capture_output=True, text=True,
                       env=env, timeout=600, cwd=ROOT)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-3000:]


@pytest.mark.parametrize("room", ["without", "between", "with"])
def test_server_admits_jobs_without_the_list(room):
    n, d, k, f, it = 300_000, 64, 600, 0.05, 5
    Xs = [synth.vmf_mixture(n, d, k, s, device="cuda") for s in (1, 2)]
    one = km.footprint(n, d, k, f, it) + 4 * n * d
    budget = {"without": one - 24 * n, "between": one - 10 * n, "with": one}[room]
    with km.Server(hbm_budget=budget, max_slots=2) as srv:
        done = [srv.wait(t) for t in [srv.submit(X, k, f, 7, 1e-6, it) for X in Xs]]
        st = srv.stats()
    assert all(s.status == 0 for s in done) and st["rejected"] == 0 and st["hbm_peak"] <= budget
    for X, s in zip(Xs, done):
        want = km.fit(X, k, f, 7, 1e-6, it)
        assert torch.equal(s.result.labels, want.labels) and s.result.J == want.J
    with km.Server(hbm_budget=one - 24 * n - (2 << 20), max_slots=1) as srv:
        with pytest.raises(km.KMeans2Error) as e:
            srv.submit(Xs[0], k, f, 7, 1e-6, it)
        assert e.value.status == -6
