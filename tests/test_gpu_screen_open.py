"""Data on which the tensor-core screen leaves most rows open (GPU): its bound grows
with ||x||^2, so a common offset in the data opens rows.  Units of 32 rows with
many open ones are decided a lane per row; results must equal the FP32 form's and
the oracle's, and a call must not cost a multiple of the FP32 form's time."""
import os
import subprocess
import sys
import time

import numpy as np
import pytest
import torch

from tests.gpu_helpers import assert_centers_close, assert_J_close, to_np

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
import paper_1108_1351_gb300 as km  # noqa: E402
from paper_1108_1351_gb300 import synth  # noqa: E402


@pytest.mark.parametrize("d", [8, 9, 11, 12, 15, 16])
@pytest.mark.parametrize("n,k", [(1, 1), (33, 2), (1025, 3), (3001, 5), (4099, 32), (3001, 33), (5003, 67),
                                 (2500, 130), (2003, 1000), (260_003, 20)])
@pytest.mark.parametrize("shift", [300.0, 1e4])
def test_steps_with_most_rows_open(n, k, d, shift):
    X = (synth.iso_gaussian_mixture(n, d, max(1, k // 2), 10 * d + k).numpy() + shift).astype(np.float32)
    rng = np.random.default_rng(n + k)
    C = X[rng.choice(n, size=k, replace=False)].astype(np.float64)
    Xd, Cd = torch.as_tensor(X, device="cuda"), torch.as_tensor(C, device="cuda")
    a, b = km.step(Xd, Cd), km.step(Xd, Cd, precision="fp32")
    assert torch.equal(a[1], b[1]) and torch.equal(a[0], b[0]) and a[2:] == b[2:]
    ocn, olab, oJ, _, oem = oracle.lloyd_step(X, C)
    assert np.array_equal(to_np(a[1]), olab)
    assert_centers_close(to_np(a[0]), ocn, X)
    assert_J_close(a[2], oJ, X)
    assert a[4] == oem


def _median_time(f):
    f()
    t = []
    for _ in range(9):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - t0)
    return sorted(t)[len(t) // 2]


@pytest.mark.parametrize("n,d,k", [(1_000_000, 16, 1000), (1_000_000, 8, 256), (4_000_000, 8, 32)])
def test_open_rows_cost_no_multiple_of_the_fp32_form(n, d, k):
    """Screen and chain together cost about 1.5 passes of the CUDA-core kernel; the
    bound leaves room for the rest of a step.  (Decided one row at a time the first
    shape took 2.3 times the FP32 form's step and 2.6 times its fit.)"""
    X = synth.iso_gaussian_mixture(n, d, k, 7, device="cuda") + 1000.0
    C = X[torch.arange(0, k, device="cuda") * (n // k)].double()
    C = km.step(X, C, precision="fp32")[0]
    auto = _median_time(lambda: km.step(X, C))
    fp32 = _median_time(lambda: km.step(X, C, precision="fp32"))
    assert auto <= 1.6 * fp32, (auto, fp32)


def _passes(f):
    a = km.screen_passes()
    r = f()
    return km.screen_passes() - a, r


@pytest.mark.parametrize("d,k", [(8, 32), (12, 20), (32, 200)])
def test_stages_leave_the_screen_where_most_rows_stay_open(d, k):
    """Every loop: queued (small stages), host-driven and graph (n k d above the
    queued loop's limit), streamed chunks and shards.  The slow stage goes on in
    the form that the fast stage ended in."""
    near = synth.iso_gaussian_mixture(200_001, d, k, 7, device="cuda")
    far = near + 1000.0
    assert _passes(lambda: km.step(near, near[:k].double()))[0] == 1
    assert _passes(lambda: km.step(near, near[:k].double(), precision="fp32"))[0] == 0
    args = (k, 0.3, 1, 1e-9, 20)
    p, r = _passes(lambda: km.fit(near, *args))
    assert p >= r.iters_fast + r.iters_slow
    assert _passes(lambda: km.fit(near, *args, precision="fp32"))[0] == 0
    assert _passes(lambda: km.fit(far, *args))[0] == 4
    p, r = _passes(lambda: km.fit_sharded(near, *args, 3))
    assert p == 3 * (r.iters_fast + r.iters_slow)
    p, r = _passes(lambda: km.fit_sharded(far, *args, 3))
    assert p == 3
    Xh = far.cpu().numpy()
    assert _passes(lambda: km.fit_streamed(Xh, *args, 50_000))[0] == 4
    p, _ = _passes(lambda: km.fit_streamed(Xh, *args, 50_000, init_centers=to_np(r.centers), start_stage=1))
    assert p == 5                                        # the five chunks of the first pass


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("far", [False, True])
def test_large_stages_decide_after_one_pass(use_graph, far):
    n, d, k = 8_000_003, 8, 32                         # n k d above the queued loop's limit
    X = synth.iso_gaussian_mixture(n, d, k, 7, device="cuda") + (1000.0 if far else 0.0)
    C = X[torch.arange(0, k, device="cuda") * (n // k)].double()
    kw = dict(init_centers=C, start_stage=1, use_graph=use_graph)
    p, got = _passes(lambda: km.fit(X, k, 0.01, 1, 0.0, 7, **kw))
    assert p == (1 if far else got.iters_slow)
    want = km.fit(X, k, 0.01, 1, 0.0, 7, precision="fp32", **kw)
    assert torch.equal(got.labels, want.labels) and torch.equal(got.centers, want.centers)
    assert (got.J, got.iters_slow) == (want.J, want.iters_slow)


BATCH = r"""
import sys, torch
sys.path.insert(0, ROOT)
import paper_1108_1351_gb300 as km
from paper_1108_1351_gb300 import synth
assert km.LIB_PATH.endswith("libkmeans2_debug.so")
jobs = [(1, 8, 1), (33, 9, 5), (1023, 16, 16), (1024, 8, 33), (1025, 12, 32), (4099, 15, 70), (6001, 16, 256),
        (5000, 24, 12)]
Xs = [synth.iso_gaussian_mixture(n, d, max(1, k // 2), j, device="cuda") + 1000.0 for j, (n, d, k) in enumerate(jobs)]
ks = [k for _, _, k in jobs]
rs, rc = km.fit_batched(Xs, ks, 0.3, list(range(len(jobs))), 1e-6, 25)
assert rc == 0
for j, (X, k, r) in enumerate(zip(Xs, ks, rs)):
    a = km.fit(X, k, 0.3, j, 1e-6, 25, precision="fp32")
    assert torch.equal(a.labels, r.labels) and torch.equal(a.centers, r.centers), jobs[j]
    assert (a.J, a.iters_fast, a.iters_slow, a.empty_clusters) == (r.J, r.iters_fast, r.iters_slow, r.empty_clusters), jobs[j]
print("ok")
"""


def test_batched_jobs_with_most_rows_open():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    from paper_1108_1351_gb300 import build
    build.build(debug=True)
    env = dict(os.environ, KMEANS2_DEBUG="1", KMEANS2_DEBUG_BATCH_POINTS="mma")
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % root + BATCH], capture_output=True,
                       text=True, env=env, timeout=600, cwd=root)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-3000:]


def test_batched_jobs_leave_the_screen():
    """A job whose first pass leaves too many rows open goes on with the CUDA-core
    kernels, the others of the batch do not: a screen that stayed would list about a
    third of the rows that the CUDA-core kernel's wider bound lists."""
    jobs = [(200_000, 8, 32), (150_001, 12, 20), (100_000, 16, 100), (200_000, 8, 32), (50_000, 24, 30), (40_000, 4, 9)]
    Xs = [synth.iso_gaussian_mixture(n, d, k, j, device="cuda") + (0.0 if j == 3 else 60.0)
          for j, (n, d, k) in enumerate(jobs)]
    Xs[0] += 60.0
    ks = [k for _, _, k in jobs]
    for _ in range(2):
        rs, rc = km.fit_batched(Xs, ks, 0.3, list(range(len(jobs))), 1e-6, 25)
        assert rc == 0
        for j, (X, k, r) in enumerate(zip(Xs, ks, rs)):
            a = km.fit(X, k, 0.3, j, 1e-6, 25, precision="fp32")
            assert torch.equal(a.labels, r.labels) and torch.equal(a.centers, r.centers), jobs[j]
            assert (a.J, a.iters_fast, a.iters_slow) == (r.J, r.iters_fast, r.iters_slow), jobs[j]
            share = r.rechecked_points / max(1, a.rechecked_points)
            if j == 0:
                assert share > 0.8, (jobs[j], share)
            if j == 3:
                assert share < 0.7, (jobs[j], share)
