"""Near ties among more centers than a warp keeps values of (1,024), GPU: one, few and
many candidates, more than the list of candidates holds (1,024), exact ties to the
lowest index, and pairs that only the oracle's order of addition ranks; few points
(a block each, up to 8,192 centers) and many (a warp each)."""
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


def _check(X, C, **kw):
    cn, lab, J, sh, em = km.step(torch.as_tensor(X, device="cuda"), torch.as_tensor(C, device="cuda"), **kw)
    ocn, olab, oJ, osh, oem = oracle.lloyd_step(X, C)
    assert np.array_equal(to_np(lab), olab)
    assert_centers_close(to_np(cn), ocn, X)
    assert_J_close(J, oJ, X)
    assert em == oem


@pytest.mark.parametrize("n", [2_000, 6_100])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 17, 33, 130])
@pytest.mark.parametrize("k", [1_025, 1_500, 8_192, 8_193])
def test_near_ties(n, d, k):
    rng = np.random.default_rng(d + k + n)
    n = max(n, k)
    C = rng.normal(size=(k, d)) * 10.0
    C[1] = C[0] + 1e-9 * rng.normal(size=d)
    C[2] = C[0]                                        # equal: lowest index
    C[3:40] = C[3] + 1e-7 * rng.normal(size=(37, d))
    C[1_000:1_025] = C[1_000] + 1e-8 * rng.normal(size=(25, d))
    X = np.concatenate([C[rng.integers(0, 40, n // 2)], C[rng.integers(0, k, n - n // 2)]])
    X = (X + 1e-3 * rng.normal(size=X.shape) * (rng.random((n, 1)) < 0.5)).astype(np.float32)
    _check(X, np.ascontiguousarray(C), precision="fp32")


@pytest.mark.parametrize("d", [2, 20, 40])
@pytest.mark.parametrize("same", [1_024, 1_025, 1_400])
def test_as_many_candidates_as_the_list_holds_and_more(d, same):
    """`same` centers at one place: all are candidates of the points there."""
    rng = np.random.default_rng(d + same)
    k = 1_500
    C = rng.normal(size=(k, d)) * 10.0
    where = rng.permutation(k)[:same]
    C[where] = 3.0
    C[where[7]] += 1e-12
    X = np.concatenate([np.full((5_500, d), 3.0), C[rng.integers(0, k, 700)]]).astype(np.float32)
    _check(X, np.ascontiguousarray(C), precision="fp32")
    X64 = X[5_000:]                                    # few points: blocks
    _check(np.ascontiguousarray(X64[:1_600] if len(X64) >= k else np.concatenate([X64] * 3)), C, precision="fp32")


def test_screened_rows_settle_among_many_centers():
    X = (synth.iso_gaussian_mixture(60_000, 17, 60, 3).numpy() + 100.0).astype(np.float32)
    C = X[np.random.default_rng(1).choice(60_000, size=1_100, replace=False)].astype(np.float64)
    Xd, Cd = torch.as_tensor(X, device="cuda"), torch.as_tensor(C, device="cuda")
    p = km.screen_passes()
    a = km.step(Xd, Cd)
    assert km.screen_passes() == p + 1
    b = km.step(Xd, Cd, precision="fp32")
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and a[2:] == b[2:]
    _check(X, C)


def test_many_ties_form_the_values_twice():
    """A point's values over all centers are formed twice, also where they are not
    kept (three or four times took 1.65 times as long here).  Against the same points
    with 1,024 centers, whose values are kept: per center no more than
    twice the time."""
    n = 300_000
    X = synth.iso_gaussian_mixture(n, 2, 50, 7, device="cuda") + 1000.0

    def per_center(k):
        C = X[torch.arange(0, k, device="cuda") * (n // k)].double().contiguous()
        km.step(X, C)
        t = []
        for _ in range(7):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            km.step(X, C)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return sorted(t)[3] / k

    assert per_center(20_000) <= 2.0 * per_center(1_024)
