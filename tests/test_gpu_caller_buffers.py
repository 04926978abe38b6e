"""Output buffers as callers hand them over (GPU): the centers may lie at any device
address, since they were always delivered by a copy.  A kernel stores them itself
only where its 8-byte stores are aligned; every other address takes the copy."""
import ctypes

import numpy as np
import pytest
import torch

import paper_1108_1351_gb300 as km
from paper_1108_1351_gb300 import binding, synth

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

N, D, K = 3_001, 8, 20


@pytest.mark.parametrize("offset", [0, 4, 8, 1])
@pytest.mark.parametrize("entry", ["step", "noalloc", "fit"])
def test_centers_out_at_any_device_address(entry, offset):
    lib = km.load()
    X = synth.iso_gaussian_mixture(N, D, K, 3, device="cuda")
    C = X[:K].double().contiguous()
    raw = torch.zeros(8 * K * D + 16, dtype=torch.uint8, device="cuda")
    lab = torch.empty(N, dtype=torch.int32, device="cuda")
    out = raw.data_ptr() + offset
    if entry == "fit":
        want = km.fit(X, K, 0.5, 1, 1e-6, 20)
        want_c, want_l = want.centers, want.labels
        rc = lib.kmeans2_fit(X.data_ptr(), N, D, K, 0.5, 1, 1e-6, 20, out, lab.data_ptr(),
                             ctypes.byref(binding.Result()), None)
    else:
        want_c, want_l = km.step(X, C)[:2]
        args = (X.data_ptr(), N, D, K, C.data_ptr(), out, lab.data_ptr(), None, None, None, None)
        rc = lib.kmeans_step(*args) if entry == "step" else lib.kmeans_step_noalloc(*args)
    assert rc == 0
    got = np.frombuffer(raw.cpu().numpy().tobytes()[offset:offset + 8 * K * D], dtype=np.float64)
    assert np.array_equal(got.reshape(K, D), want_c.cpu().numpy())
    assert torch.equal(lab, want_l)
    rest = raw.cpu().numpy()
    assert not rest[:offset].any() and not rest[offset + 8 * K * D:].any()
