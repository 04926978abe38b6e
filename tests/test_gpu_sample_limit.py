"""The draws at the number of keys (n + m) up to which one CTA makes them (GPU)."""
import numpy as np
import pytest
import torch

from tests.gpu_helpers import to_np

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
import paper_1108_1351_gb300 as km  # noqa: E402


@pytest.mark.parametrize("n,k,f", [(60_000, 7, 1.0), (60_001, 7, 1.0), (60_000, 300, 1.0), (60_001, 300, 1.0),
                                   (119_993, 7, 1e-5), (119_994, 7, 1e-5), (100_000, 5_000, 0.2),
                                   (100_001, 5_000, 0.2)])
def test_draws_at_the_limit(n, k, f):
    sub, pos = km.sample(n, k, f, 5, device="cuda")
    osub, opos = oracle.sample(n, k, f, 5)
    assert np.array_equal(to_np(sub), osub) and np.array_equal(to_np(pos), opos)


def test_many_keys_are_not_left_to_one_cta():
    """130,000 keys: one CTA took 308 us where the grid takes 300.  Counted by
    launches: the grid's selection is some 35 of them, one CTA's is one."""
    X = torch.randn(65_000, 2, device="cuda")

    def launches(rows):
        p = km.Profile()
        r = km.fit(X[:rows], 3, 1.0, 1, 1e-6, 1, profile=p)
        assert r.iters_fast == r.iters_slow == 1
        return p.kernel_launches

    assert launches(65_000) >= launches(50_000) + 20
