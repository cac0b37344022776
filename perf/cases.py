"""The calls whose speed is measured: whole clustering jobs, batches, a served mix and the
no-allocation nearest-center pass, each through the binding a user's program calls.

``listed()`` names the fixed cases, ``draw(rng)`` gives one more of the same ranges,
``prepare(case, seed)`` makes what a program holds before the call (points, handles),
``run(state)`` is one pass with its results, ``work(case)`` the bytes and operations the
pass cannot do without and ``exact(case, seed)`` the results in float64 from plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1412_1947_gb300 import binding as B

DEV = "cuda"
FP32, TC = "fp32", "tc"
DIMS = (2, 3, 4, 5, 7, 8, 10, 13, 16, 16, 20, 24, 32, 32, 33, 48, 64, 64, 100, 128, 128)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: labels and SSE of a few points against few centers, for a host
        # that cannot allocate device memory; a launch and little else
        {"name": "assign-small", "kind": "assign", "n": 1000, "d": 16, "k": 16},
        # the same call on a whole dataset with many centers (1 M odd rows, d = 64)
        {"name": "assign-large", "kind": "assign", "n": 1000003, "d": 64, "k": 300},
        # the small configuration: 4096 points, 3 blobs, 16 subclusters, default options;
        # launches and latency
        {"name": "job-small", "kind": "job", "n": 4096, "d": 4, "N": 256, "local_k": 16, "final_k": 3, "iters": 20,
         "prec": FP32, "graph": False, "host": False, "bf16": False, "blobs": 3, "outliers": 0.0},
        # the paper's timing data: 2-D, 500 points per blob, compression 10 (many rounds,
        # 500 final centers), recorded once and replayed
        {"name": "job-2d", "kind": "job", "n": 250000, "d": 2, "N": 1000, "local_k": 100, "final_k": 500, "iters": 25,
         "prec": FP32, "graph": True, "host": False, "bf16": False, "blobs": 500, "outliers": 0.0},
        # a table of measurements handed over as a numpy array, odd in every size (the
        # Seeds data's 7 attributes), default options; uploads its points on every pass
        {"name": "job-odd-host", "kind": "job", "n": 200003, "d": 7, "N": 2001, "local_k": 40, "final_k": 77,
         "iters": 25, "prec": FP32, "graph": False, "host": True, "bf16": False, "blobs": 77, "outliers": 0.01},
        # the headline workload: 2^20 x 16, 256 subclusters of 4096, 64 centers each
        {"name": "job-headline", "kind": "job", "n": 1 << 20, "d": 16, "N": 4096, "local_k": 64, "final_k": 64,
         "iters": 25, "prec": TC, "graph": True, "host": False, "bf16": False, "blobs": 64, "outliers": 0.01},
        # one job of the serving stream by itself: bfloat16 storage, the widest rows
        {"name": "job-bf16-d128", "kind": "job", "n": 400000, "d": 128, "N": 6250, "local_k": 25, "final_k": 300,
         "iters": 25, "prec": TC, "graph": False, "host": False, "bf16": True, "blobs": 300, "outliers": 0.0},
        # Algorithm 2's uneven subclusters in place of the peel
        {"name": "job-unequal", "kind": "unequal", "n": 500009, "d": 32, "m": 128, "local_k": 32, "final_k": 100,
         "iters": 25, "prec": TC, "blobs": 100},
        # many tiny independent problems at once, an odd width
        {"name": "batch-small", "kind": "batch", "count": 300, "shape": 1, "d": 5, "lo": 40, "hi": 600, "per_k": 32,
         "min_k": 3, "iters": 20, "prec": FP32},
        # the uneven batch: 2048 instances of 256 .. 65536 rows
        {"name": "batch-uneven", "kind": "batch", "count": 2048, "shape": 2, "d": 32, "lo": 256, "hi": 65536,
         "per_k": 256, "min_k": 8, "iters": 25, "prec": TC},
        # a burst of served jobs of mixed sizes, widths and storage types (the serving
        # workload's stream), four slots
        {"name": "serve-mix", "kind": "serve", "count": 20, "shape": 3, "n_lo": 10000, "n_hi": 1000000, "slots": 4,
         "prec": TC},
        # the largest: 2^24 x 64, 1024 blobs, 256 local and 1024 final centers
        {"name": "job-large", "kind": "job", "n": 1 << 24, "d": 64, "N": 65536, "local_k": 256, "final_k": 1024,
         "iters": 25, "prec": TC, "graph": True, "host": False, "bf16": False, "blobs": 1024, "outliers": 0.0},
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.999))))


def draw(rng):
    kind = rng.choice(("assign", "job", "job", "job", "job", "unequal", "batch", "serve"))
    d = rng.choice(DIMS)
    if kind == "assign":
        n, k = _log_int(rng, 1000, 2000000), _log_int(rng, 2, 1024)
        while n * k * d > 4e10:
            n, k = n // 2 + 1, max(2, k // 2)
        return {"kind": kind, "n": n, "d": d, "k": k}
    if kind == "batch":
        lo, per_k = _log_int(rng, 32, 256), rng.choice((16, 32, 100, 256))
        case = {"kind": kind, "count": _log_int(rng, 10, 1000), "shape": rng.randrange(1 << 20), "d": d, "lo": lo,
                "hi": lo * _log_int(rng, 2, 50), "per_k": per_k, "min_k": rng.choice((3, 8)),
                "iters": rng.choice((10, 20, 25)), "prec": rng.choice((FP32, TC))}
        while case["count"] > 4 and work(case)["flops"] > 1e11:
            case["count"] = case["count"] * 2 // 3
        return case
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(6, 20), "shape": rng.randrange(1 << 20), "n_lo": 10000,
                "n_hi": _log_int(rng, 50000, 1000000), "slots": rng.randint(2, 6), "prec": rng.choice((FP32, TC, TC))}
    n = _log_int(rng, 1000, 4000000)
    while n * d > 1 << 26:
        n = n // 2 + 1
    N = max(n // 400 + 1, _log_int(rng, 200, max(201, n // 4)))
    local_k = min(N, max(4, min(256, N // rng.choice((5, 16, 64, 128)))))
    iters, prec = rng.choice((10, 20, 25)), rng.choice((FP32, TC, TC))
    while n * local_k * iters * d > (1e12 if prec == TC and d in (16, 32, 64) else 5e10):
        local_k = local_k // 2 + 1
    final_k = min(_log_int(rng, 3, 1024), -(-n // N) * local_k // 2 + 1)
    case = {"kind": kind, "n": n, "d": d, "local_k": local_k, "final_k": final_k, "iters": iters, "prec": prec,
            "blobs": max(2, min(final_k, 1024))}
    if kind == "unequal":
        case["m"] = max(2, min(512, n // N))
        case["final_k"] = min(final_k, local_k)        # some of the m groups may stay empty
        return case
    case.update({"N": N, "graph": rng.random() < 0.5, "host": rng.random() < 0.2, "bf16": rng.random() < 0.25,
                 "outliers": rng.choice((0.0, 0.01))})
    return case


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _mixture(n, d, blobs, g, outliers=0.0):
    """n x d float32 points: isotropic Gaussians (means in [0, 10]^d, sigma in [0.2, 1]),
    a share of them uniform outliers instead."""
    means = torch.rand((blobs, d), generator=g, device=DEV) * 10.0
    sig = 0.2 + 0.8 * torch.rand(blobs, generator=g, device=DEV)
    which = torch.randint(0, blobs, (n,), generator=g, device=DEV)
    out = torch.empty((n, d), device=DEV)
    step = max(1, (1 << 26) // d)
    for a in range(0, n, step):
        b = min(n, a + step)
        w = which[a:b]
        torch.randn((b - a, d), generator=g, device=DEV, out=out[a:b])
        out[a:b].mul_(sig[w][:, None]).add_(means[w])
    if outliers:
        rows = torch.randperm(n, generator=g, device=DEV)[:int(outliers * n)]
        out[rows] = torch.rand((len(rows), d), generator=g, device=DEV) * 16.0 - 3.0
    return out


def _job_points(case, seed):
    x = _mixture(case["n"], case["d"], case["blobs"], _gen(seed), case.get("outliers", 0.0))
    return x.to(torch.bfloat16) if case.get("bf16") else x


def _batch_shape(case):
    """Sizes and center counts of the instances (the case's own, whatever the seed)."""
    r = np.random.default_rng(case["shape"])
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    sizes = np.floor(np.exp(r.uniform(lo, hi, size=case["count"]))).astype(np.int64)
    return sizes, np.maximum(case["min_k"], sizes // case["per_k"]).astype(np.int32)


def _batch_points(case, seed):
    """One mixture per instance, k blobs each."""
    sizes, k = _batch_shape(case)
    g = _gen(seed)
    rows, d = int(sizes.sum()), case["d"]
    total = int(k.sum())
    means = torch.rand((total, d), generator=g, device=DEV) * 10.0
    sig = 0.2 + 0.8 * torch.rand(total, generator=g, device=DEV)
    first = torch.from_numpy(np.cumsum(k) - k).to(DEV)
    s, kk = torch.from_numpy(sizes).to(DEV), torch.from_numpy(k.astype(np.int64)).to(DEV)
    inst = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), s)
    blob = first[inst] + (torch.rand(rows, generator=g, device=DEV) * kk[inst]).long().clamp_(max=kk[inst] - 1)
    return torch.randn((rows, d), generator=g, device=DEV).mul_(sig[blob][:, None]).add_(means[blob]), sizes, k


def _serve_jobs(case, seed):
    """Job shapes of the serving stream: N = ceil(n / 64), local centers by subcluster size
    and final k, half the jobs in bfloat16."""
    r = np.random.default_rng(case["shape"])
    jobs = []
    for i in range(case["count"]):
        n = int(math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        d = int(r.choice((8, 32, 128)))
        fk = int(math.exp(r.uniform(math.log(8), math.log(1024))))
        N = -(-n // 64)
        S = -(-n // N)
        lk = min(N, max(8, -(-N // 256), -(-2 * fk // S)))
        jobs.append({"n": n, "d": d, "N": N, "local_k": lk, "final_k": min(fk, S * lk), "iters": 25,
                     "blobs": max(2, fk), "bf16": bool(r.random() < 0.5), "prec": case["prec"], "seed": int(seed) + i})
    return jobs


class _State:
    """What a program keeps: inputs and the library's handles, given back at the end."""

    def __init__(self, **kw):
        self.__dict__.update(kw)

    def __del__(self):
        for h in ("job", "batch", "server"):
            if self.__dict__.get(h) is not None:
                self.__dict__[h].close()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "assign":
        n, d, k = case["n"], case["d"], case["k"]
        x = _mixture(n, d, k, _gen(seed))
        x = (x - x.amin(0)) / (x.amax(0) - x.amin(0))
        c = x[torch.randint(0, n, (k,), generator=_gen(seed + 1), device=DEV)].contiguous()
        return _State(case=case, x=x, c=c, labels=torch.empty(n, dtype=torch.int32, device=DEV),
                      sse=torch.empty(1, dtype=torch.float64, device=DEV))
    if kind == "batch":
        x, sizes, k = _batch_points(case, seed)
        torch.cuda.synchronize()
        return _State(case=case, batch=B.Batch(x, sizes, k), seed=int(seed), prec=B.PRECISIONS[case["prec"]])
    if kind == "serve":
        jobs = _serve_jobs(case, seed)
        pts = [_job_points(j, j["seed"]) for j in jobs]
        torch.cuda.synchronize()
        return _State(case=case, jobs=jobs, pts=pts, prec=B.PRECISIONS[case["prec"]],
                      server=B.Server(slots=case["slots"], hbm_budget_bytes=40 * 10**9))
    x = _job_points(case, seed)
    if case.get("host"):
        x = x.cpu().view(torch.int16).numpy().view(np.uint16) if case["bf16"] else x.cpu().numpy()
    torch.cuda.synchronize()
    job = B.Job(x)
    if case.get("graph"):
        job.option(B.PSCL_OPT_GRAPH, 1)
    return _State(case=case, x=x, job=job, seed=int(seed), prec=B.PRECISIONS[case["prec"]])


# ------------------------------------------------------------------ one pass
def run(state):
    case, kind = state.case, state.case["kind"]
    if kind == "assign":
        B.pscl_assign_sse_noalloc(state.x, state.c, state.labels, state.sse, torch.cuda.current_stream().cuda_stream)
        return {"labels": state.labels, "sse": state.sse}
    if kind == "batch":
        state.batch.run(case["iters"], state.seed, state.prec)
        centers, labels, sse = state.batch.result()
        return {"centers": centers, "labels": labels, "sse": sse}
    if kind == "serve":
        s = state.server
        tickets = [s.submit(x, j["N"], j["local_k"], j["final_k"], j["iters"], j["seed"], state.prec, want_labels=True)
                   for j, x in zip(state.jobs, state.pts)]
        out = []
        for t in tickets:
            s.wait(t)
            centers, labels, sse, _ = s.fetch(t)
            out.append({"centers": centers, "labels": labels, "sse": sse})
        return out
    job = state.job
    job.load(state.x)
    if kind == "unequal":
        job.steps_unequal(case["m"], case["local_k"], case["final_k"], case["iters"], state.seed, state.prec)
    else:
        job.run(case["N"], case["local_k"], case["final_k"], case["iters"], state.seed, state.prec)
    centers, labels, sse = job.result()
    return {"centers": centers, "labels": labels, "sse": sse}


# ------------------------------------------------------------------ what a pass cannot do without
def _job_evals(c):
    """Distance evaluations of a job: local and final Lloyd, and the nearest final center."""
    n = c["n"]
    S = c["m"] if c["kind"] == "unequal" else -(-n // c["N"])
    P = min(S * c["local_k"], n)
    return (n * c["local_k"] + P * c["final_k"]) * c["iters"] + n * c["final_k"]


def work(case):
    kind, d = case["kind"], case.get("d")
    if kind == "assign":
        n, k = case["n"], case["k"]
        return {"bytes": n * d * 4 + k * d * 4 + n * 4 + 8, "flops": 2.0 * n * k * d}
    if kind == "batch":
        sizes, k = _batch_shape(case)
        k = np.minimum(k, sizes)
        rows = int(sizes.sum())
        return {"bytes": rows * d * 4 + rows * 4 + int(k.sum()) * d * 4 + 8 * len(sizes),
                "flops": 2.0 * d * float((sizes * k).sum()) * (case["iters"] + 1)}
    if kind == "serve":
        parts = [work({**j, "kind": "job"}) for j in _serve_jobs(case, 0)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    n = case["n"]
    return {"bytes": n * d * (2 if case.get("bf16") else 4) + n * 4 + case["final_k"] * d * 4 + 8,
            "flops": 2.0 * d * _job_evals(case)}


# ------------------------------------------------------------------ the results in 64 bits
_M64 = (1 << 64) - 1


def _splitmix(s):
    s = (s + 0x9E3779B97F4A7C15) & _M64
    z = s
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return s, z ^ (z >> 31)


def _first_members(m, k, seed, stage, index):
    """The first k entries of the seeded Fisher-Yates shuffle of 0 .. m-1."""
    _, key = _splitmix((stage << 32) | index)
    s, at = (seed ^ key) & _M64, {}
    for i in range(k):
        s, r = _splitmix(s)
        j = i + r % (m - i)
        at[i], at[j] = at.get(j, j), at.get(i, i)
    return torch.tensor([at[i] for i in range(k)], device=DEV)


def _nearest(x, c):
    """(index, squared distance) of each row's nearest center."""
    lab = torch.empty(len(x), dtype=torch.long, device=DEV)
    step = max(1, (1 << 27) // len(c))
    c2 = (c * c).sum(1)
    for a in range(0, len(x), step):
        lab[a:a + step] = (c2 - 2.0 * (x[a:a + step] @ c.T)).argmin(1)
    dist = torch.empty(len(x), dtype=torch.float64, device=DEV)
    for a in range(0, len(x), 1 << 20):
        t = x[a:a + (1 << 20)] - c[lab[a:a + (1 << 20)]]
        dist[a:a + (1 << 20)] = (t * t).sum(1)
    return lab, dist


def _lloyd(x, k, iters, seed, stage, index):
    k = min(k, len(x))
    c = x[_first_members(len(x), k, seed, stage, index)].clone()
    for _ in range(iters):
        lab = (((c * c).sum(1) - 2.0 * (x @ c.T)).argmin(1))
        cnt = torch.bincount(lab, minlength=k)
        tot = torch.zeros_like(c).index_add_(0, lab, x)
        c = torch.where(cnt[:, None] > 0, tot / cnt.clamp(min=1)[:, None], c)
    return c


def _scaled(x, bf16=False):
    """Min-max scaling in float64, rounded to the storage type as the method defines."""
    x = x.double()
    lo, hi = x.amin(0), x.amax(0)
    y = torch.where(hi > lo, (x - lo) * (1.0 / (hi - lo)), torch.zeros_like(x))
    return y.to(torch.bfloat16 if bf16 else torch.float32).double()


def _peel(x, N):
    left, out = torch.arange(len(x), device=DEV), []
    while len(left) > N:
        rows = x[left]
        key = ((rows - rows.amin(0)) ** 2).sum(1)
        order = torch.sort(key, stable=True).indices
        out.append(left[order[:N].sort().values])
        left = left[order[N:].sort().values]
    return out + [left]


def _groups(x, m):
    lo, hi = x.amin(0), x.amax(0)
    t = (torch.arange(m, device=DEV, dtype=torch.float64) + 0.5) / m
    lm = (lo + t[:, None] * (hi - lo)).float().double()
    g, _ = _nearest(x, lm)
    order = torch.sort(g, stable=True).indices
    return [p for p in torch.split(order, torch.bincount(g, minlength=m).tolist()) if len(p)]


def _two_level(case, seed, points):
    x = _scaled(points, case.get("bf16", False))
    parts = _groups(x, case["m"]) if case["kind"] == "unequal" else _peel(x, case["N"])
    pool = torch.cat([_lloyd(x[p], case["local_k"], case["iters"], seed, 0, i) for i, p in enumerate(parts)])
    c = _lloyd(pool, case["final_k"], case["iters"], seed, 1, 0)
    return {"centers": c.cpu().numpy(), "labels": None, "sse": float(_nearest(x, c)[1].sum())}


def exact(case, seed):
    kind, seed = case["kind"], int(seed)
    if work(case)["flops"] > 4e12:
        return None
    if kind == "assign":
        s = prepare(case, seed)
        return {"labels": None, "sse": _nearest(s.x.double(), s.c.double())[1].sum().reshape(1)}
    if kind == "batch":
        if case["count"] > 1000:
            return None
        x, sizes, k = _batch_points(case, seed)
        centers, sse, at = [], [], 0
        for i, m in enumerate(sizes):
            y = _scaled(x[at:at + int(m)])
            at += int(m)
            c = _lloyd(y, int(k[i]), case["iters"], seed, 0, i)
            centers.append(c)
            sse.append(_nearest(y, c)[1].sum())
        return {"centers": torch.cat(centers).cpu().numpy(), "labels": None, "sse": torch.stack(sse).cpu().numpy()}
    if kind == "serve":
        return [_two_level({**j, "kind": "job"}, j["seed"], _job_points(j, j["seed"])) for j in _serve_jobs(case, seed)]
    return _two_level(case, seed, _job_points(case, seed))
