"""The work that is timed: what callers of the k-means library have it do.

Each case is one call (or, for the server, one burst of requests) through the
package's public entry points at the library's defaults.  Inputs come from
the package's own generators (``synth``); sizes from the workloads of
``bench.py`` and the tests, scaled where noted so that one pass takes
milliseconds to a few hundred milliseconds.

Kinds of case:
  step     km.step: one Lloyd iteration from given centers
  noalloc  km.step_noalloc: the same from the library's fixed scratch
  fit      km.fit: the whole two-stage method
  batched  km.fit_batched: many uneven independent fits in one call
  serve    km.Server: a burst of jobs of different n, d, k on several slots
  streamed km.fit_streamed: data that stays in page-locked host memory
"""
import math

import numpy as np
import torch

import paper_1108_1351_gb300 as km
from paper_1108_1351_gb300 import synth

DEV = "cuda"


def listed():
    return [
        # the smallest workload (20,000 points in the plane, 4 clusters): one
        # iteration, where launches, allocations and waits are all the time
        dict(name="step_gauss2d", kind="step", gen="iso", n=20_000, d=2, k=4),
        # one iteration inside a loop that must not allocate; odd n and d
        dict(name="noalloc_d5", kind="noalloc", gen="iso", n=262_147, d=5, k=50),
        # one iteration at a ragged middle dimension (no vector width divides it)
        dict(name="step_d37", kind="step", gen="iso", n=200_003, d=37, k=100),
        # one iteration on embedding-like data: 16-bit tensor-core form (split)
        dict(name="step_vmf128", kind="step", gen="vmf", n=500_000, d=128, k=1024),
        # the smallest workload as a whole fit, sampling included
        dict(name="fit_gauss2d", kind="fit", gen="iso", n=20_000, d=2, k=4, f=0.1, tol=1e-6,
             max_iter=100, least=2),
        # the paper's 10-million-point shape (12 dimensions)
        dict(name="fit_d12", kind="fit", gen="iso", n=10_000_000, d=12, k=16, f=0.1, tol=1e-6,
             max_iter=100, least=2),
        # the large-scale workload (anisotropic clusters with noise, 1 % subset)
        # at a fifth of its size; runs to max_iter in both stages
        dict(name="fit_aniso8", kind="fit", gen="aniso", n=100_000_000, d=8, k=32, f=0.01,
             tol=1e-5, max_iter=50, least=50),
        # a serving-sized request: wide points, few clusters
        dict(name="fit_d128_k32", kind="fit", gen="iso", n=300_000, d=128, k=32, f=0.1, tol=1e-6,
             max_iter=100, least=2),
        # the embedding workload (d = 128, k = 1024) at a fiftieth of its size
        dict(name="fit_vmf128", kind="fit", gen="vmf", n=1_000_000, d=128, k=1024, f=0.02,
             tol=1e-6, max_iter=50, least=10),
        # 64 of the batched workload's instances: n 1e3..1e6, d in {2, 8, 32, 64}, k 2..256
        dict(name="batched_64", kind="batched", count=64, f=0.1, tol=1e-6, max_iter=100, least=2),
        # ten requests of the serving workload (n up to 500,000) on 4 slots
        dict(name="serve_10", kind="serve", count=10, n_hi=500_000, k_hi=512, slots=4, f=0.1,
             tol=1e-6, max_iter=100, least=2),
        # the large-scale workload's shape with X left in host memory
        dict(name="streamed_d8", kind="streamed", gen="aniso", n=10_000_000, d=8, k=32, f=0.01,
             tol=1e-5, max_iter=50, least=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds; sizes log-uniform over their ranges,
    the work per pass at most the largest listed case's."""
    kind = rng.choice(["step", "step", "noalloc", "fit", "fit", "fit", "batched", "serve",
                       "streamed"])
    if kind in ("step", "noalloc"):
        d = rng.choice([2, 3, 5, 8, 12, 16, 23, 32, 37, 64, 100, 128])
        k = _log_int(rng, 2, 1024)
        n = _log_int(rng, 20_000, min(4_194_304, 4e10 / (d * k)))
        gen = "vmf" if d >= 64 and k >= 64 else "iso"
        return dict(kind=kind, gen=gen, n=max(n, k), d=d, k=k)
    if kind == "fit":
        d = rng.choice([2, 3, 4, 7, 8, 12, 16, 31, 32, 64, 128])
        k = _log_int(rng, 2, 1024)
        n = _log_int(rng, 20_000, min(1e7, 4e10 / (d * k)))
        gen = "vmf" if d >= 64 and k >= 64 else ("aniso" if d == 8 else "iso")
        return dict(kind=kind, gen=gen, n=max(n, k), d=d, k=k, f=rng.choice([0.01, 0.02, 0.1, 0.3]),
                    tol=rng.choice([1e-3, 1e-5, 1e-6]), max_iter=rng.choice([20, 50]), least=2)
    if kind == "batched":
        return dict(kind=kind, count=_log_int(rng, 8, 48), f=0.1, tol=1e-6, max_iter=100, least=2)
    if kind == "serve":
        return dict(kind=kind, count=rng.randint(4, 10), n_hi=500_000, k_hi=512,
                    slots=rng.choice([1, 2, 4, 8]), f=0.1, tol=1e-6, max_iter=100, least=2)
    d = rng.choice([4, 8, 12])
    return dict(kind=kind, gen="aniso", n=_log_int(rng, 100_000, 8e7 / d), d=d,
                k=_log_int(rng, 4, 64), f=0.01, tol=1e-5, max_iter=rng.choice([20, 50]), least=2)


def _points(gen, n, d, k, seed):
    if gen == "vmf":
        return synth.vmf_mixture(n, d, k, seed, device=DEV)
    if gen == "aniso":
        return synth.aniso_gaussian_noise(n, d, k, seed, device=DEV)
    return synth.iso_gaussian_mixture(n, d, k, seed, device=DEV)


def _jobs(case, seed):
    """(n, d, k, seed) of each job of a batched or serve case."""
    base = seed * 100_003
    if case["kind"] == "batched":
        # the workload's first instances: the sizes belong to the case, the points to the seed
        return [(s.n, s.d, s.k, base + i)
                for i, s in enumerate(synth.instance_specs(case["count"], seed=0))]
    trace = synth.arrival_trace(200.0, 10.0, 1, n_hi=case["n_hi"], k_hi=case["k_hi"])
    return [(j.n, j.d, j.k, base + i) for i, j in enumerate(trace[:case["count"]])]


def _job_points(n, d, k, seed):
    return synth.iso_gaussian_mixture(n, d, k, seed, lo=-20.0, hi=20.0, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind, "seed": seed}
    if kind in ("batched", "serve"):
        st["jobs"] = _jobs(case, seed)
        st["X"] = [_job_points(*j) for j in st["jobs"]]
        if kind == "serve":
            st["server"] = km.Server(max_slots=case["slots"])
    else:
        X = _points(case["gen"], case["n"], case["d"], case["k"], seed)
        if kind in ("step", "noalloc"):
            # the centers a run is at: some points, moved a little
            rows = torch.from_numpy(np.random.default_rng(seed + 1).choice(
                case["n"], size=case["k"], replace=False)).to(X.device)
            st["C"] = (X[rows].double() * 0.95).contiguous()
        if kind == "streamed":
            X = X.cpu().pin_memory()
        st["X"] = X
    torch.cuda.synchronize()
    return st


def _fit_out(r):
    return dict(centers=r.centers, labels=r.labels, J=r.J, shift_fast=r.shift_fast,
                shift_slow=r.shift_slow, iters_fast=r.iters_fast, iters_slow=r.iters_slow,
                converged=[int(r.converged_fast), int(r.converged_slow)],
                empty_clusters=r.empty_clusters, subset_size=r.subset_size)


def _all_out(rs):
    """The results of several jobs, joined: one tensor or array per field."""
    num = {f: np.array([getattr(r, f) for r in rs])
           for f in ("J", "shift_fast", "shift_slow", "iters_fast", "iters_slow",
                     "converged_fast", "converged_slow", "empty_clusters", "subset_size")}
    return dict(centers=torch.cat([r.centers.reshape(-1) for r in rs]),
                labels=torch.cat([r.labels for r in rs]), **num)


def run(state):
    case, kind, X = state["case"], state["kind"], state["X"]
    if kind == "step":
        return list(km.step(X, state["C"]))
    if kind == "noalloc":
        return list(km.step_noalloc(X, state["C"]))
    seed = state["seed"]
    if kind == "fit":
        return _fit_out(km.fit(X, case["k"], case["f"], seed, case["tol"], case["max_iter"]))
    if kind == "streamed":
        return _fit_out(km.fit_streamed(X, case["k"], case["f"], seed, case["tol"],
                                        case["max_iter"], 0))
    jobs = state["jobs"]
    if kind == "batched":
        rs, _ = km.fit_batched(X, [j[2] for j in jobs], case["f"], [j[3] for j in jobs],
                               case["tol"], case["max_iter"])
        return _all_out(rs)
    srv = state["server"]
    tickets = [srv.submit(x, j[2], case["f"], j[3], case["tol"], case["max_iter"])
               for x, j in zip(X, jobs)]
    done = [srv.wait(t) for t in tickets]
    return _all_out([s.result for s in done])


def work(case):
    """One read of X (and of given centers), one write of labels and centers;
    2 d flop per distance, over one iteration (step) or over the `least`
    iterations a stage takes (every listed fit takes at least that many)."""
    def one(n, d, k, centers_in, evals):
        return 4 * n * d + 4 * n + 8 * k * d * (2 if centers_in else 1), 2 * d * evals

    if case["kind"] in ("step", "noalloc"):
        b, f = one(case["n"], case["d"], case["k"], True, case["n"] * case["k"])
        return {"bytes": b, "flops": f}
    jobs = _jobs(case, 0) if case["kind"] in ("batched", "serve") else \
        [(case["n"], case["d"], case["k"], 0)]
    tb = tf = 0
    for n, d, k, _ in jobs:
        m = min(n, max(k, math.ceil(case["f"] * n)))
        b, f = one(n, d, k, False, case["least"] * k * (m + n))
        tb, tf = tb + b, tf + f
    return {"bytes": tb, "flops": tf}


# ---------------------------------------------------------------- 64-bit values

def _step64(X, C, chunk):
    """One Lloyd iteration in FP64: new centers, labels, J, shift, empty."""
    n, (k, d) = X.shape[0], C.shape
    cn = (C * C).sum(1)
    labels = torch.empty(n, dtype=torch.int32, device=X.device)
    S = torch.zeros_like(C)
    N = torch.zeros(k, dtype=torch.float64, device=X.device)
    J = torch.zeros((), dtype=torch.float64, device=X.device)
    for a in range(0, n, chunk):
        x = X[a:a + chunk].to(C.device).double()
        lab = torch.addmm(cn, x, C.t(), alpha=-2.0).argmin(1)
        J += ((x - C[lab]) ** 2).sum()
        labels[a:a + chunk] = lab
        if k * d <= 1024:       # few targets: a product instead of colliding atomic adds
            hot = torch.nn.functional.one_hot(lab, k).double()
            S += hot.t() @ x
            N += hot.sum(0)
        else:
            S.index_add_(0, lab, x)
            N += torch.bincount(lab, minlength=k)
    new = torch.where(N[:, None] > 0, S / N.clamp(min=1.0)[:, None], C)
    shift = float(((new - C) ** 2).sum(1).max().sqrt())
    return new, labels, float(J), shift, int((N == 0).sum())


_M64 = (1 << 64) - 1


def _keys(seed, first, count):
    """SplitMix64 outputs of stream positions [first, first + count)."""
    with np.errstate(over="ignore"):
        i = np.arange(count, dtype=np.uint64) + np.uint64((first + 1) & _M64)
        z = np.uint64(seed & _M64) + i * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _fit64(X, k, f, seed, tol, max_iter):
    n, d = X.shape
    m = min(n, max(k, math.ceil(f * n)))
    keys = _keys(seed, 0, n)
    sub = np.sort(np.argpartition(keys, m - 1)[:m]) if m < n else np.arange(n)
    kc = _keys(seed, n, m)
    first = np.argpartition(kc, k - 1)[:k] if k < m else np.arange(m)
    pos = first[np.argsort(kc[first])]
    Xs = X[torch.from_numpy(sub).to(X.device)].to(DEV)
    C = Xs[torch.from_numpy(pos).to(DEV)].double()
    chunk = max(1024, int(2 ** 26 // max(k, d)))
    out = {}
    for stage, P in (("fast", Xs), ("slow", X)):
        it, conv = 0, False
        while it < max_iter and not conv:
            C, lab, J, shift, empty = _step64(P, C, chunk)
            it += 1
            conv = shift <= tol
        out[stage] = (it, int(conv), shift)
    return dict(centers=C, labels=lab, J=J, shift_fast=out["fast"][2], shift_slow=out["slow"][2],
                iters_fast=out["fast"][0], iters_slow=out["slow"][0],
                converged=[out["fast"][1], out["slow"][1]], empty_clusters=empty, subset_size=m)


def exact(case, seed):
    st_kind = case["kind"]
    if st_kind in ("step", "noalloc"):
        st = prepare(case, seed)
        return list(_step64(st["X"], st["C"], max(1024, int(2 ** 26 // max(case["k"], case["d"])))))
    if st_kind in ("fit", "streamed"):
        n, d, k = case["n"], case["d"], case["k"]
        if n * (1.0 + case["f"]) * k * d * case["max_iter"] > 2e12:
            return None
        X = _points(case["gen"], n, d, k, seed)
        return _fit64(X, k, case["f"], seed, case["tol"], case["max_iter"])
    jobs = _jobs(case, seed)
    if sum(n * (1.0 + case["f"]) * k * d for n, d, k, _ in jobs) * case["max_iter"] > 2e12:
        return None
    rs = [_fit64(_job_points(n, d, k, s), k, case["f"], s, case["tol"], case["max_iter"])
          for n, d, k, s in jobs]
    out = {f: np.array([r[f] for r in rs])
           for f in ("J", "shift_fast", "shift_slow", "iters_fast", "iters_slow")}
    for i, f in enumerate(("converged_fast", "converged_slow")):
        out[f] = np.array([bool(r["converged"][i]) for r in rs])
    out["empty_clusters"] = np.array([r["empty_clusters"] for r in rs])
    out["subset_size"] = np.array([r["subset_size"] for r in rs])
    return dict(centers=torch.cat([r["centers"].reshape(-1) for r in rs]),
                labels=torch.cat([r["labels"] for r in rs]), **out)
