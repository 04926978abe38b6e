"""The three loops that run a stage's iterations (GPU): queued ahead of the
read-back (small stages), as a while-graph, and one round trip per iteration.

Which one runs depends on the work of an iteration, so a child process with the
debug library (device index checks on) takes KMEANS2_DEBUG_QUEUED_WORK to send small
data through each of them: queued to the end, queued and then as a graph, graph,
and host-driven.  Every loop must give the oracle's labels and iteration counts
and the same centers, J and trajectories bit for bit, with the CUDA-core kernel, the
screen, and a screen that the stage leaves; stages end at and next to the ends of
the queued chunks (4, 12, 28) and of the queued part before a graph (12)."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASE = r"""
import os, sys
import numpy as np, torch
sys.path.insert(0, ROOT)
import oracle
import paper_1108_1351_gb300 as km
from paper_1108_1351_gb300 import synth
assert km.LIB_PATH.endswith("libkmeans2_debug.so")
LOOPS = {"queued": (None, False), "queued, graph": (None, True), "graph": ("-1", True), "host": ("-1", False)}

def run(loop, f):
    env, graph = LOOPS[loop]
    os.environ.pop("KMEANS2_DEBUG_QUEUED_WORK", None)
    if env:
        os.environ["KMEANS2_DEBUG_QUEUED_WORK"] = env
    p0 = km.screen_passes()
    r = f(graph)
    return r, km.screen_passes() - p0

def key(r):
    return (r.J, r.iters_fast, r.iters_slow, r.converged_fast, r.converged_slow, r.shift_fast, r.shift_slow,
            r.empty_clusters) + tuple(t.tobytes() for _, t in sorted(r.traj.items()))

def chunks(iters, most):
    q, c = 0, 4
    while q < iters:
        q += min(c, most - q)
        c = min(2 * c, 32)
    return q

for n, d, k, far in DATA:
    X = (synth.aniso_gaussian_noise(n, d, k, d).numpy() + far).astype(np.float32)
    Xd = torch.as_tensor(X, device="cuda")
    C = X[np.random.default_rng(d).choice(n, size=k, replace=False)].astype(np.float64)
    # tolerances that end the slow stage at (or before) the iterations asked for
    t = km.fit(Xd, k, 0.5, 3, 0.0, 60, init_centers=C, start_stage=1, trajectories=True, precision="fp32").traj
    shifts = [float(v) for v in t["shift_slow"]]
    ends = [(0.0, m) for m in (1, 3, 4, 5, 12, 13, 27, 28, 29, 36, 60)]
    ends += [(min(shifts[:i]), 60) for i in (3, 4, 5, 11, 12, 13, 28, 29) if i <= len(shifts)]
    for tol, most in ends:
        want = next((i + 1 for i, s in enumerate(shifts[:most]) if s <= tol), min(most, len(shifts)))
        first = None
        for loop in LOOPS:
            r, passes = run(loop, lambda g: km.fit(Xd, k, 0.5, 3, tol, most, init_centers=C, start_stage=1,
                                                   use_graph=g, trajectories=True))
            assert r.iters_slow == want, (d, loop, tol, most, r.iters_slow, want)
            if first is None:
                first = r
            assert key(r) == key(first), (d, loop, tol, most)
            assert torch.equal(r.labels, first.labels) and torch.equal(r.centers, first.centers), (d, loop, tol, most)
            # the kernel that ran
            if d < 8:
                assert passes == 0
            elif far:
                assert passes == (1 if loop in ("graph", "host") or most == 1 else min(4, most)), (d, loop, passes)
            elif loop == "queued":
                assert passes == chunks(want, most), (d, loop, most, want, passes)
            elif loop == "queued, graph" and most >= 36:
                assert passes == (chunks(want, 12) if want <= 12 else want), (d, loop, most, want, passes)
            elif loop in ("graph", "host"):
                assert passes == want, (d, loop, passes, want)
    # both stages against the oracle
    for most in (5, 13, 40):
        o = oracle.fit(X, k, 0.3, 5, 1e-6, most)
        for loop in LOOPS:
            r, _ = run(loop, lambda g: km.fit(Xd, k, 0.3, 5, 1e-6, most, use_graph=g, trajectories=True))
            assert np.array_equal(r.labels.cpu().numpy(), o["labels"]), (d, loop, most)
            assert (r.iters_fast, r.iters_slow) == (o["iters_fast"], o["iters_slow"]), (d, loop, most)
            assert abs(r.J - o["J"]) <= 1e-9 * o["J"], (d, loop, most)
print("ok")
"""

DATA = [(6_001, 3, 7, 0.0), (6_001, 8, 12, 0.0), (4_001, 12, 33, 0.0), (3_001, 40, 20, 0.0), (6_001, 8, 12, 1000.0)]


def test_every_stage_loop_gives_the_same_fit():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1108_1351_gb300 import build
    build.build(debug=True)
    env = dict(os.environ, KMEANS2_DEBUG="1")
    env.pop("KMEANS2_DEBUG_QUEUED_WORK", None)
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\nDATA = %r\n" % (ROOT, DATA) + CASE],
                       capture_output=True, text=True, env=env, timeout=900, cwd=ROOT)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-3000:]
