"""The work that users of this framework have it do, as measured cases.

Every case is one pass through the public Python API (``paper_2406_06488_gb300.ept``):
a single permutation test on host arrays or on CUDA tensors, the same test on the
caller's own relabelings, a batched run of many tests, a burst of served requests, and
a test in the streaming mode.  Sizes are the named workloads of this repository, the
paper's experiment sizes, or generic odd ones.  The samples always differ a little (a
mean shift or a larger variance), or in a batch every other test does, as in the
repository's workloads.
"""
import math
import random

import numpy as np
import torch

from paper_2406_06488_gb300 import ept

# what a program reads from a result: the statistic of the samples, the permuted
# statistics and the p-value with the count behind it


def listed():
    return [
        # the interactive call: a hundred rows a side in numpy arrays; launches and latency
        dict(name="small_host", kind="single", where="host", stat="ed", nx=100, ny=100, p=10, B=1000, mean=0.2,
             var=1.0),
        # the paper's experiment size (nx = ny = 200, p = 500, B = 200), data already on the GPU
        dict(name="paper_size", kind="single", where="device", stat="ed", nx=200, ny=200, p=500, B=200, mean=0.05,
             var=1.0),
        # an ordinary test with no round size anywhere
        dict(name="ragged", kind="single", where="device", stat="ed", nx=777, ny=1333, p=333, B=4999, mean=0.03,
             var=1.0),
        # the headline workload: many features, a small shift, 10^4 permutations
        dict(name="highdim", kind="single", where="device", stat="ed", nx=2000, ny=3000, p=1000, B=10000, mean=0.01,
             var=1.0),
        # the large kernel test (Gaussian MMD, 10^4 rows a side)
        dict(name="mmd", kind="single", where="device", stat="mmd", nx=10000, ny=10000, p=100, B=10000, mean=0.0,
             var=1.1),
        # a small treated group against many controls, Laplacian kernel
        dict(name="unequal_laplace", kind="single", where="device", stat="mmd_laplace", nx=9001, ny=499, p=257,
             B=5000, mean=0.05, var=1.0),
        # bandwidth unknown: the median heuristic, host arrays in, host statistics out
        dict(name="median_host", kind="median", where="host", stat="mmd", nx=6000, ny=4500, p=64, B=2000, mean=0.02,
             var=1.0),
        # restricted permutations (within strata) supplied by the caller as bit masks
        dict(name="caller_masks", kind="masks", where="device", stat="ed", nx=1500, ny=1100, p=50, B=5000, mean=0.05,
             var=1.0),
        # a simulation study: 500 replications of the paper's null experiment in one run
        dict(name="replications", kind="batch", tests=500, n_lo=200, n_hi=200, p_lo=100, p_hi=100, B=200, mean=0.1,
             mix=0),
        # a screening run: 512 uneven tests in one run
        dict(name="batch_uneven", kind="batch", tests=512, n_lo=50, n_hi=2000, p_lo=20, p_hi=500, B=5000, mean=0.1,
             mix=1),
        # a burst of requests to the serving scheduler, all submitted and then collected
        dict(name="serving_burst", kind="serving", tests=16, n_lo=100, n_hi=6000, p_lo=10, p_hi=1000, B=5000,
             mean=0.05, mix=2),
        # blocks larger than the memory the context may take: windows of row panels
        dict(name="stream", kind="stream", where="device", stat="ed", nx=50000, ny=50000, p=64, B=4000, mean=0.01,
             var=1.0, budget_gb=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "median", "masks", "batch", "batch", "serving", "stream"])
    if kind == "batch":
        lo = _log_int(rng, 20, 400)
        hi = _log_int(rng, lo, 1600)
        tests = max(2, min(_log_int(rng, 8, 500), int(2.0e9 / (4.0 * hi * hi * 100))))
        return dict(kind="batch", tests=tests, n_lo=lo, n_hi=hi, p_lo=_log_int(rng, 5, 60), p_hi=_log_int(rng, 60, 400),
                    B=_log_int(rng, 99, 3000), mean=0.1, mix=rng.randrange(1 << 20))
    if kind == "serving":
        return dict(kind="serving", tests=rng.randint(3, 20), n_lo=50, n_hi=_log_int(rng, 500, 5000), p_lo=10,
                    p_hi=_log_int(rng, 50, 800), B=_log_int(rng, 500, 5000), mean=0.05, mix=rng.randrange(1 << 20))
    if kind == "stream":
        n = _log_int(rng, 30000, 70000)
        nx = int(n * rng.uniform(0.3, 0.7))
        return dict(kind="stream", where=rng.choice(["device", "host"]), stat="ed", nx=nx, ny=n - nx,
                    p=rng.randint(8, 96), B=_log_int(rng, 500, 3000), mean=0.01, var=1.0,
                    budget_gb=round(2.0 * n * n / 2.0 ** 30 * rng.uniform(0.3, 0.8), 2))
    hi = 20000 if kind == "single" else 9000
    n = _log_int(rng, 60, hi)
    share = rng.choice([0.5, rng.uniform(0.3, 0.7), rng.uniform(0.03, 0.3)])
    nx = max(2, int(n * share))
    if rng.random() < 0.5:
        nx = n - nx
    p = min(_log_int(rng, 3, 1500), max(3, int(1.2e7 / n)))
    B = _log_int(rng, 99, 10000)
    stat = "mmd" if kind == "median" else rng.choice(["ed", "ed", "mmd", "mmd_laplace"])
    # relabelings are drawn on the GPU here, so a test that uses them has everything there
    return dict(kind=kind, where="device" if kind == "masks" else rng.choice(["device", "host"]), stat=stat, nx=nx, ny=n - nx, p=p, B=B,
                mean=round(rng.uniform(0.02, 0.2), 3), var=1.0)


def _shapes(case):
    """The tests of a batch or burst: sizes, statistic and permutation count of each."""
    r = random.Random(case["mix"])
    out = []
    for t in range(case["tests"]):
        if case["kind"] == "serving":   # as the serving workload: sizes log-uniform, ED and MMD mixed
            nx, ny = _log_int(r, case["n_lo"], case["n_hi"]), _log_int(r, case["n_lo"], case["n_hi"])
            p, stat = _log_int(r, case["p_lo"], case["p_hi"]), r.choice(["ed", "mmd"])
            B, mean = r.choice([max(1, case["B"] // 5), case["B"], 4 * case["B"]]), case["mean"]
        else:                           # as the batched workload: sizes uniform, every other test null
            nx, ny = r.randint(case["n_lo"], case["n_hi"]), r.randint(case["n_lo"], case["n_hi"])
            p, stat, B = r.randint(case["p_lo"], case["p_hi"]), "ed", case["B"]
            mean = case["mean"] if t % 2 else 0.0
        out.append(dict(nx=nx, ny=ny, p=p, stat=stat, B=B, mean=mean, var=1.0, test=t))
    return out


def _sigma(stat, p):
    return 1.0 if stat == "ed" else math.sqrt(p)


def _samples(c, seed, host):
    """X ~ N(0, I) and Y ~ N(mean, var I), from the seed alone."""
    key = 1_000_003 * seed + c.get("test", 0)
    if host:
        r = np.random.default_rng(key)
        X = r.standard_normal((c["nx"], c["p"]), dtype=np.float32)
        Y = r.standard_normal((c["ny"], c["p"]), dtype=np.float32)
        Y = Y * np.float32(math.sqrt(c["var"])) + np.float32(c["mean"])
        return X, Y
    g = torch.Generator(device="cuda").manual_seed(key)
    X = torch.randn(c["nx"], c["p"], device="cuda", generator=g)
    Y = torch.randn(c["ny"], c["p"], device="cuda", generator=g) * math.sqrt(c["var"]) + c["mean"]
    return X, Y


def _masks(case, seed):
    """Relabelings that permute within four strata of the pooled rows (row t belongs to
    stratum t mod 4): bit t % 32 of word t // 32 is set where row t goes to x*."""
    nx, n, B = case["nx"], case["nx"] + case["ny"], case["B"]
    g = torch.Generator(device="cuda").manual_seed(1_000_003 * seed + 77)
    member = torch.zeros(B, (n + 31) // 32 * 32, dtype=torch.bool, device="cuda")
    for k in range(4):
        rows = torch.arange(k, n, 4, device="cuda")
        mx = int((rows < nx).sum())
        pick = torch.rand(B, rows.numel(), device="cuda", generator=g).argsort(dim=1)[:, :mx]
        member[torch.arange(B, device="cuda")[:, None], rows[pick]] = True
    bits = member.view(B, -1, 32).to(torch.int64) << torch.arange(32, device="cuda")
    words = bits.sum(dim=2)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32), member[:, :n]


def prepare(case, seed):
    """The samples where the program has them, and the context it keeps."""
    kind = case["kind"]
    if kind in ("batch", "serving"):
        tests = []
        for c in _shapes(case):
            X, Y = _samples(c, seed, kind == "serving")
            tests.append(dict(X=X, Y=Y, B=c["B"], seed=seed + c["test"], stat=c["stat"], sigma=_sigma(c["stat"], c["p"])))
        if kind == "serving":
            return dict(ctx=ept.Context(0), kind=kind, tests=tests)
        ctx = ept.Context(0)
        return dict(ctx=ctx, kind=kind, batch=ctx.prepare_batch(tests))
    X, Y = _samples(case, seed, case["where"] == "host")
    budget = int(case["budget_gb"] * 2 ** 30) if kind == "stream" else 0
    s = dict(ctx=ept.Context(0, budget_bytes=budget), kind=kind, X=X, Y=Y,
             args=dict(stat=case["stat"], sigma="median" if kind == "median" else _sigma(case["stat"], case["p"])))
    if kind == "masks":
        s["masks"] = _masks(case, seed)[0]
    else:
        s["args"].update(B=case["B"], seed=seed)
    return s


def _answer(r):
    return dict(observed=r.observed, p_value=r.p_value, n_ge=r.n_ge, sigma=r.sigma, stats=r.stats)


def _answers(rs):
    cat = torch.cat if isinstance(rs[0].stats, torch.Tensor) else np.concatenate
    return dict(observed=np.array([r.observed for r in rs]), p_value=np.array([r.p_value for r in rs]),
                n_ge=np.array([r.n_ge for r in rs]), stats=cat([r.stats for r in rs]))


def run(state):
    ctx, kind = state["ctx"], state["kind"]
    if kind == "batch":
        return _answers(state["batch"].run())
    if kind == "serving":
        tickets = [ctx.submit(**t) for t in state["tests"]]
        return _answers([ctx.wait(t) for t in tickets])
    if kind == "masks":
        return _answer(ctx.test_masks(state["X"], state["Y"], state["masks"], **state["args"]))
    return _answer(ctx.test(state["X"], state["Y"], **state["args"]))


def work(case):
    """Samples (and caller's masks) read, statistics written; 2 p operations for each of
    the n(n+1)/2 distinct pairs and 2 for each pair and relabeling."""
    b = f = 0.0
    for c in (_shapes(case) if case["kind"] in ("batch", "serving") else [case]):
        n = c["nx"] + c["ny"]
        b += 4.0 * n * c["p"] + 8.0 * c["B"]
        if case["kind"] == "masks":
            b += c["B"] * ((n + 31) // 32) * 4.0
        f += n * (n + 1.0) * (c["p"] + c["B"] + 1.0)
    return dict(bytes=b, flops=f)


# ---- the same results in 64 bits, from the definitions ----
_M32 = 0xFFFFFFFF


def _philox(c0, blo, bhi, klo, khi):
    """Philox4x32-10 of counters (c0, 0, blo, bhi) under keys (klo, khi), unsigned 32-bit
    words in int64 tensors; the two 64-bit output words as (high, low) halves."""
    x0, x1, x2, x3 = c0, torch.zeros_like(c0), blo, bhi
    for _ in range(10):
        p0, p1 = x0 * 0xD2511F53, x2 * 0xCD9E8D57   # low 64 bits of the products
        x0, x1, x2, x3 = ((p1 >> 32) & _M32) ^ x1 ^ klo, p1 & _M32, ((p0 >> 32) & _M32) ^ x3 ^ khi, p0 & _M32
        klo, khi = (klo + 0x9E3779B9) & _M32, (khi + 0xBB67AE85) & _M32
    return (x1, x0), (x3, x2)


def _relabelings(nx, n, B, seeds):
    """Draws 1..B of the permutation streams of some tests of one shape: uint8
    [n, tests * B], 1 where the pooled row goes to x* (selection sampling)."""
    dev = "cuda"
    b = torch.arange(1, B + 1, dtype=torch.int64, device=dev).repeat(len(seeds))[None, :]
    s = torch.tensor(seeds, dtype=torch.int64, device=dev).repeat_interleave(B)[None, :]
    need = torch.full((b.shape[1],), nx, dtype=torch.int64, device=dev)
    out = torch.empty(n, b.shape[1], dtype=torch.uint8, device=dev)
    step = max(2, min(512, int(2e7 // b.shape[1]) // 2 * 2))
    for t0 in range(0, n, step):
        t1 = min(n, t0 + step)
        c0 = torch.arange(t0 // 2, (t1 + 1) // 2, dtype=torch.int64, device=dev)[:, None].expand(-1, b.shape[1])
        z = torch.zeros_like(c0)
        words = _philox(c0, z + (b & _M32), z + (b >> 32), s & _M32, (s >> 32) & _M32)
        for t in range(t0, t1):
            hi, lo = words[t & 1][0][(t - t0) // 2], words[t & 1][1][(t - t0) // 2]
            rank = (hi * (n - t) + ((lo * (n - t)) >> 32)) >> 32
            keep = rank < need
            need = need - keep.to(torch.int64)
            out[t] = keep
    return out


def _pooled(X, Y, stat, sigma):
    """The pooled n x n matrix of distances or kernel values, and the bandwidth."""
    Z = torch.cat([torch.as_tensor(X, device="cuda"), torch.as_tensor(Y, device="cuda")]).double()
    D = torch.cdist(Z, Z, compute_mode="donot_use_mm_for_euclid_dist")
    if stat == "ed":
        return D, 0.0
    if sigma == "median":
        n = D.shape[0]
        d = torch.cat([D[i, i + 1:] for i in range(n)]).sort().values
        sigma = float(d[(d.numel() - 1) // 2])
    if stat == "mmd":
        return torch.exp(D * D / (-2.0 * sigma * sigma)), sigma
    return torch.exp(-D / sigma), sigma


def _statistics(W, member, nx, ny, stat):
    """Eq. 1 / Eq. 2 for the columns of member [n, columns] (1: the row is in x*)."""
    out, L1, S = [], W.sum(dim=1), float(W.sum())
    for j in range(0, member.shape[1], 2048):
        s = member[:, j:j + 2048].double()
        xx = (s * (W @ s)).sum(dim=0)
        L = L1 @ s
        v = 2.0 / (nx * ny) * (L - xx) - xx / (nx * nx) - (S - 2.0 * L + xx) / (ny * ny)
        out.append(v if stat == "ed" else -v)
    return torch.cat(out)


def _exact_test(X, Y, stat, sigma, member):
    nx, n = X.shape[0], X.shape[0] + Y.shape[0]
    W, sig = _pooled(X, Y, stat, sigma)
    own = (torch.arange(n, device="cuda") < nx).to(torch.uint8)[:, None]
    v = _statistics(W, torch.cat([own, member], dim=1), nx, n - nx, stat)
    obs, stats = float(v[0]), v[1:]
    ge = int((stats >= obs).sum())
    return dict(observed=obs, p_value=(1.0 + ge) / (1.0 + stats.numel()), n_ge=ge, sigma=sig, stats=stats)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serving"):
        shapes = _shapes(case)
        if work(case)["flops"] > 4e12:   # minutes in 64 bits
            return None
        groups, res = {}, [None] * len(shapes)
        for c in shapes:
            groups.setdefault((c["nx"], c["ny"], c["B"]), []).append(c)
        for (nx, ny, B), cs in groups.items():
            member = _relabelings(nx, nx + ny, B, [seed + c["test"] for c in cs])
            for k, c in enumerate(cs):
                X, Y = _samples(c, seed, kind == "serving")
                res[c["test"]] = _exact_test(X, Y, c["stat"], _sigma(c["stat"], c["p"]), member[:, k * B:(k + 1) * B])
        stats = torch.cat([r["stats"] for r in res])
        return dict(observed=np.array([r["observed"] for r in res]), p_value=np.array([r["p_value"] for r in res]),
                    n_ge=np.array([r["n_ge"] for r in res]), stats=stats.cpu().numpy() if kind == "serving" else stats)
    n = case["nx"] + case["ny"]
    if n > 25000:                        # the pooled matrix alone is 80 GB at the listed size
        return None
    X, Y = _samples(case, seed, case["where"] == "host")
    if kind == "masks":
        member = _masks(case, seed)[1].T.to(torch.uint8)
    else:
        member = _relabelings(case["nx"], n, case["B"], [seed])
    r = _exact_test(X, Y, case["stat"], "median" if kind == "median" else _sigma(case["stat"], case["p"]), member)
    if case["where"] == "host":
        r["stats"] = r["stats"].cpu().numpy()
    return r
