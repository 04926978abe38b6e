"""The kernels that start and finish an iteration (GPU): the stage start (centers
spread over warps and CTAs, padding), the exact sum of squares, and the update
with its 192-by-32-bit divisions and its last-CTA reduction.  Center counts lie
around 8 per CTA, 256 per reduction pass, 1024 per reduction round and the cap
of 1024 CTAs; data reach the ends of the fixed-point range."""
import numpy as np
import pytest
import torch

from tests.gpu_helpers import assert_centers_close, assert_J_close, to_np

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
import paper_1108_1351_gb300 as km  # noqa: E402


def _check(X, C):
    cn, lab, J, sh, em = km.step(torch.as_tensor(X, device="cuda"), torch.as_tensor(C, device="cuda"),
                                 precision="fp32")
    ocn, olab, oJ, osh, oem = oracle.lloyd_step(X, C)
    assert np.array_equal(to_np(lab), olab)
    assert_centers_close(to_np(cn), ocn, X)
    assert_J_close(J, oJ, X)
    assert abs(sh - osh) <= 1e-10 * max(osh, 1.0)
    assert em == oem


@pytest.mark.parametrize("k", [1, 7, 8, 9, 255, 256, 257, 1023, 1025, 2049, 8200])
@pytest.mark.parametrize("d", [1, 5, 33])
def test_center_counts(k, d):
    rng = np.random.default_rng(k + d)
    X = rng.normal(size=(2 * k + 37, d)).astype(np.float32) * 3.0
    C = X[rng.choice(X.shape[0], size=k, replace=False)].astype(np.float64)
    _check(X, C)


@pytest.mark.parametrize("case", ["powers", "wide", "negative", "ties_of_the_grid", "constant"])
def test_value_ranges(case):
    rng = np.random.default_rng(3)
    X = rng.normal(size=(5003, 6)).astype(np.float32)
    if case == "powers":                      # at and next to powers of two, both signs
        e = rng.integers(-3, 10, size=X.shape).astype(np.float64)
        X = np.ldexp(1.0, e.astype(int)).astype(np.float32) * np.sign(X)
        X[0, 0] = np.nextafter(np.float32(1024.0), np.float32(0))
    elif case == "wide":                      # within the 2^23 below the largest value
        X = (X * np.exp(rng.uniform(-8, 6, size=X.shape))).astype(np.float32)
    elif case == "negative":
        X = (-np.abs(X) - 100.0).astype(np.float32)
    elif case == "ties_of_the_grid":          # halves of the low part's unit
        X = (rng.integers(-2 ** 22, 2 ** 22, size=X.shape) + 0.5).astype(np.float32)
    else:
        X[:] = np.float32(0.1)
    C = X[rng.choice(X.shape[0], size=11, replace=False)].astype(np.float64)
    _check(X, C)


@pytest.mark.parametrize("d", [16, 17, 32, 33, 64, 128, 300])
@pytest.mark.parametrize("k", [2, 33, 130, 256, 700])
def test_recheck_forms(d, k):
    """Near ties of every kind: one, two and many candidates, exact ties and
    pairs that only the oracle's order of addition can rank."""
    rng = np.random.default_rng(d + k)
    C = rng.normal(size=(k, d))
    C[1] = C[0] + 1e-9 * rng.normal(size=d)
    if k > 2:
        C[2] = C[0]                                   # equal: lowest index
        C[3:20] = C[3] + 1e-7 * rng.normal(size=(17, d))
    X = np.concatenate([C[rng.integers(0, k, 600)], 0.5 * (C[0] + C[rng.integers(0, k, 600)])])
    X = (X + 1e-3 * rng.normal(size=X.shape) * (rng.random((X.shape[0], 1)) < 0.5)).astype(np.float32)
    _check(X, np.ascontiguousarray(C))


@pytest.mark.parametrize("chunk", [0, 4_000, 2_001, 1_999, 700, 1_000_000])
def test_streamed_chunk_orders(chunk):
    """One, two, odd and even chunk counts, ragged last chunks: passes alternate
    their direction and reuse the chunks still in the buffers."""
    from paper_1108_1351_gb300 import synth
    X = synth.aniso_gaussian_noise(4_001, 8, 12, 4).numpy()
    o = oracle.fit(X, 12, 0.1, 3, 1e-6, 40)
    s = km.fit_streamed(X, 12, 0.1, 3, 1e-6, 40, chunk)
    r = km.fit(torch.as_tensor(X, device="cuda"), 12, 0.1, 3, 1e-6, 40)
    assert np.array_equal(to_np(s.labels), o["labels"])
    assert np.array_equal(to_np(s.centers), to_np(r.centers)) and s.J == r.J
    assert (s.iters_fast, s.iters_slow) == (o["iters_fast"], o["iters_slow"])


def _same(a, b):
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and a[2:] == b[2:]


@pytest.mark.parametrize("precision", ["bf16", "fp16"])
@pytest.mark.parametrize("n,d,k", [(1, 16, 1), (33, 16, 3), (5003, 48, 4), (20_001, 128, 130),
                                   (9_000, 32, 4096), (9_000, 32, 4097)])
def test_moved_row_sums(precision, n, d, k):
    """First and later passes of the 16-bit forms, whose moved rows are listed and
    added by cluster: up to the largest k of the list and past it, runs of one
    cluster and of many, and passes that move few rows or none."""
    rng = np.random.default_rng(n + k)
    X = (rng.normal(size=(n, d)) + 4.0 * rng.integers(0, 3, size=(n, 1))).astype(np.float32)
    C = X[rng.integers(0, n, size=k)].astype(np.float64)
    C[: k // 2] += 50.0                               # clusters that no row joins
    Xd = torch.as_tensor(X, device="cuda")
    Cd = torch.as_tensor(C, device="cuda")
    _same(km.step(Xd, Cd, precision=precision), km.step(Xd, Cd, precision="fp32"))
    if k <= n // 8:
        f = km.fit(Xd, k, 0.3, 1, 1e-7, 60, precision=precision)
        g = km.fit(Xd, k, 0.3, 1, 1e-7, 60, precision="fp32")
        assert torch.equal(f.labels, g.labels) and torch.equal(f.centers, g.centers)
        assert f.J == g.J and f.iters_slow == g.iters_slow


def test_moved_rows_past_the_list():
    """More moved rows than the list holds (2^22): the distance kernel adds the rest."""
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(4_500_000, 16, device="cuda", generator=g)
    C = X[:40].double().contiguous()
    _same(km.step(X, C, precision="bf16"), km.step(X, C, precision="fp32"))


@pytest.mark.parametrize("n,k,f", [(9_000, 256, 0.5), (9_000, 257, 0.5), (9_000, 5_000, 1.0),
                                   (65_536, 300, 1.0), (65_537, 300, 1.0), (131_071, 7, 1e-5),
                                   (131_072, 7, 1e-5), (400, 400, 1.0), (1, 1, 1.0)])
def test_draws_around_the_one_cta_limits(n, k, f):
    sub, pos = km.sample(n, k, f, 11, device="cuda")
    osub, opos = oracle.sample(n, k, f, 11)
    assert np.array_equal(to_np(sub), osub) and np.array_equal(to_np(pos), opos)
