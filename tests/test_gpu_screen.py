"""The tensor-core screen of the FP32 form (precision AUTO, 8 <= d <= 128; GPU).

The screen decides a row only outside its bound and leaves the others to the
FP32 chain and the FP64 recheck, so labels, centers, J and iteration counts
must equal the oracle's (labels exactly; centers and J within the helpers'
derived tolerances) and the plain FP32 form's bit for bit.  Sizes lie around
the edges of its tiles: 32 / 64 rows per warp and 256 to 512 per step, 8 centers per
block, 16 / 32 per chunk, d at, between and outside the padded sizes 8 .. 128."""
import os
import subprocess
import sys

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

DEV = "cuda"


def _check_step(X, C):
    Xd, Cd = torch.as_tensor(X, device=DEV), torch.as_tensor(C, device=DEV)
    a = km.step(Xd, Cd)
    b = km.step(Xd, Cd, precision="fp32")
    assert torch.equal(a[1], b[1]) and torch.equal(a[0], b[0]) and a[2:] == b[2:]
    ocn, olab, oJ, _, oem = oracle.lloyd_step(X, C)
    assert np.array_equal(to_np(a[1]), olab)
    assert_centers_close(to_np(a[0]), ocn, X)
    assert_J_close(a[2], oJ, X)
    assert a[4] == oem


@pytest.mark.parametrize("d", [7, 8, 9, 12, 16, 17, 32, 33, 48, 50, 64, 65, 96, 100, 128, 129])
@pytest.mark.parametrize("n,k", [(1, 1), (31, 7), (64, 8), (65, 9), (511, 16), (513, 17),
                                 (2000, 33), (5000, 257), (3000, 1000), (170_003, 20)])
def test_step_sizes(n, k, d):
    X = synth.iso_gaussian_mixture(n, d, max(1, k // 2), 100 * d + k).numpy()
    rng = np.random.default_rng(n + k)
    C = X[rng.choice(n, size=k, replace=False)].astype(np.float64)
    _check_step(X, C)


@pytest.mark.parametrize("d", [8, 40])
@pytest.mark.parametrize("scale,shift", [(1e-20, 0.0), (1e-12, 0.0), (1e6, 0.0), (1.0, 1e4)])
def test_step_ranges(scale, shift, d):
    X = (synth.iso_gaussian_mixture(3001, d, 9, 5).numpy() * scale + shift).astype(np.float32)
    _check_step(X, X[:20].astype(np.float64))


@pytest.mark.parametrize("d", [8, 16, 24, 100])
def test_step_centers_outside_the_scaled_range_and_duplicates(d):
    X = synth.iso_gaussian_mixture(1500, d, 5, 6).numpy()
    C = X[:40].astype(np.float64)
    C[3] *= 1e14                       # far beyond the FP16 scaling: every row goes to the FP32 chain
    _check_step(X, C)
    C = np.concatenate([X[:20], X[:20]]).astype(np.float64)     # exact ties: lowest index
    _check_step(X, C)
    _check_step(np.ascontiguousarray(np.repeat(X[:50], 30, axis=0)), X[:33].astype(np.float64))


@pytest.mark.parametrize("n,d,k", [(20_011, 9, 4), (60_001, 8, 32), (30_003, 12, 50),
                                   (20_003, 31, 70), (9_001, 100, 20)])
def test_fits_and_other_entry_points(n, d, k):
    X = synth.aniso_gaussian_noise(n, d, k, d).numpy()
    Xd = torch.as_tensor(X, device=DEV)
    a = km.fit(Xd, k, 0.1, 3, 1e-6, 40)
    b = km.fit(Xd, k, 0.1, 3, 1e-6, 40, precision="fp32")
    assert a.precision_used == b.precision_used == "fp32"
    same = (lambda r: (r.J, r.iters_fast, r.iters_slow, r.shift_slow, r.empty_clusters))
    assert torch.equal(a.labels, b.labels) and torch.equal(a.centers, b.centers) and same(a) == same(b)
    o = oracle.fit(X, k, 0.1, 3, 1e-6, 40)
    assert np.array_equal(to_np(a.labels), o["labels"])
    assert (a.iters_fast, a.iters_slow) == (o["iters_fast"], o["iters_slow"])
    s = km.fit_streamed(X, k, 0.1, 3, 1e-6, 40, 7_001)
    assert np.array_equal(to_np(s.labels), o["labels"]) and s.J == a.J
    h = km.fit_sharded(Xd, k, 0.1, 3, 1e-6, 40, 3)
    assert torch.equal(h.labels, a.labels) and torch.equal(h.centers, a.centers) and h.J == a.J
    C = Xd[:k].double()
    p, q = km.step_noalloc(Xd, C), km.step(Xd, C, precision="fp32")
    assert torch.equal(p[1], q[1]) and torch.equal(p[0], q[0]) and p[2:] == q[2:]


BATCH = r"""
import sys, torch
sys.path.insert(0, ROOT)
import paper_1108_1351_gb300 as km
from paper_1108_1351_gb300 import synth
assert km.LIB_PATH.endswith("libkmeans2_debug.so")
jobs = [(1, 8, 1), (33, 9, 5), (1023, 16, 16), (1024, 8, 33), (1025, 17, 32), (4099, 31, 70),
        (6001, 32, 256), (5000, 33, 12), (3001, 50, 100), (7003, 64, 200), (2500, 7, 20), (2049, 2, 9)]
Xs = [synth.aniso_gaussian_noise(n, d, max(2, k // 2), 7 + j, device="cuda") if n > 40 else
      synth.iso_gaussian_mixture(n, d, 1, j, device="cuda") for j, (n, d, k) in enumerate(jobs)]
ks = [k for _, _, k in jobs]
rs, rc = km.fit_batched(Xs, ks, 0.3, list(range(len(jobs))), 1e-6, 25)
assert rc == 0
for j, (X, k, r) in enumerate(zip(Xs, ks, rs)):
    a = km.fit(X, k, 0.3, j, 1e-6, 25, precision="fp32")
    assert torch.equal(a.labels, r.labels) and torch.equal(a.centers, r.centers), jobs[j]
    assert (a.J, a.iters_fast, a.iters_slow, a.empty_clusters) == (r.J, r.iters_fast, r.iters_slow, r.empty_clusters), jobs[j]
print("ok")
"""


def test_batched_screen_equals_single_fits():
    """The batched form with the screen forced on every job it may take (debug
    build, device index checks on): items of 1,024 rows and their remainders,
    every dimension class, k at the chunk edges."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    from paper_1108_1351_gb300 import build
    build.build(debug=True)
    env = dict(os.environ, KMEANS2_DEBUG="1", KMEANS2_DEBUG_BATCH_POINTS="mma")
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % root + BATCH], capture_output=True,
                       text=True, env=env, timeout=600, cwd=root)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-3000:]
