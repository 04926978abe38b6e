"""The update's grid (GPU): one CTA up to 8 centers, then one center per CTA up to
152 CTAs, then warps and threads of a CTA that take several."""
import numpy as np
import pytest
import torch

from tests.gpu_helpers import assert_centers_close, assert_J_close, to_np

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
import paper_1108_1351_gb300 as km  # noqa: E402


@pytest.mark.parametrize("d", [2, 40])
@pytest.mark.parametrize("k", [8, 9, 151, 152, 153, 304, 305, 1216, 1217, 10_001])
def test_center_counts_at_the_grid(k, d):
    rng = np.random.default_rng(k)
    X = rng.normal(size=(k + 700, d)).astype(np.float32) * 3.0
    C = X[rng.choice(X.shape[0], size=k, replace=False)].astype(np.float64)
    cn, lab, J, sh, em = km.step(torch.as_tensor(X, device="cuda"), torch.as_tensor(C, device="cuda"))
    ocn, olab, oJ, osh, oem = oracle.lloyd_step(X, C)
    assert np.array_equal(to_np(lab), olab)
    assert_centers_close(to_np(cn), ocn, X)
    assert_J_close(J, oJ, X)
    assert abs(sh - osh) <= 1e-10 * max(osh, 1.0) and em == oem
