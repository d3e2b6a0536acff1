"""Cases that time the ZipLine search through its public entry points, over the range of shapes it is used on.

A case names an entry point, an objective, a cluster recipe, the shape ([B] instances of n workers x R predicted
iterations) and whether the rows are verified to be sorted:

  select    ``ZipLine.select_batched``          timestamps on the GPU, results on the GPU
  predict   ``ZipLine.predict_select_batched``  last end timestamps and intervals on the GPU; both phases in one call
  host      ``ZipLine.select_batched_host``     timestamps and results in pinned host memory, copies included
  noalloc   ``zl_select_batched_noalloc``       no handle, scratch fixed inside the library

The recipes are the heterogeneous clusters that the repository's configurations describe (see ``RECIPES``); inputs are
int64 microseconds, made on the GPU from the seed.  Results are whole numbers, so every comparison is exact.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2001_01347_b200 as zl

# mean iteration time of a worker (microseconds), how means spread over the workers, jitter of one iteration
RECIPES = {
    # workers of one kind with a moderate spread
    "lognormal": dict(mean=200_000.0, sigma=0.3, jitter=0.05),
    # nearly homogeneous workers, one in ten three times slower
    "stragglers": dict(mean=150_000.0, sigma=0.2, jitter=0.10, slow_share=0.10, slow_by=3.0),
    # widely spread workers, one iteration in a hundred takes five times as long
    "spiky": dict(mean=100_000.0, sigma=0.5, jitter=0.08, spike_share=0.01, spike_by=5.0),
    # two generations of machines, started within a second of each other
    "bimodal": dict(mean=80_000.0, second=240_000.0, sigma=0.0, jitter=0.05, offset=1_000_000.0),
}
OBJECTIVES = {"range": zl.ZL_OBJ_RANGE, "sum": zl.ZL_OBJ_SUM}


def _case(name, entry, objective, recipe, n, R, B, checked=False):
    return {"name": name, "entry": entry, "objective": objective, "recipe": recipe, "n": n, "R": R, "B": B, "checked": checked}


def listed():
    return [
        # one decision for a handful of workers, the search every barrier of a small training job makes: pure latency
        _case("range_n4_R8_B1", "select", "range", "lognormal", 4, 8, 1),
        # one decision for a large cluster (largest shape of the paper's Table II)
        _case("range_n1000_R150_B1", "select", "range", "lognormal", 1000, 150, 1),
        # the same for the total-wait objective at the table's middle shape
        _case("sum_n100_R150_B1", "select", "sum", "lognormal", 100, 150, 1),
        # a scheduler that weighs thousands of small what-if scenarios in one call
        _case("range_n16_R64_B4096", "select", "range", "lognormal", 16, 64, 4096),
        # a thousand mid-size jobs with stragglers
        _case("range_n128_R256_B1024", "select", "range", "stragglers", 128, 256, 1024),
        # the headline workload: 64 large clusters with heavy-tailed iterations
        _case("range_n1024_R1024_B64", "select", "range", "spiky", 1024, 1024, 64),
        # the largest instances: long look-ahead on a cluster of two machine generations
        _case("range_n4096_R4096_B8", "select", "range", "bimodal", 4096, 4096, 8),
        # the headline workload under the total-wait objective: a full merge, nothing can be skipped
        _case("sum_n1024_R1024_B64", "select", "sum", "spiky", 1024, 1024, 64),
        # a ragged batch from an untrusted source: odd sizes, rows verified on the way
        _case("range_n93_R211_B257_checked", "select", "range", "stragglers", 93, 211, 257, True),
        # both phases in one call: the matrix of predictions never exists
        _case("predict_n1024_R1024_B64", "predict", "range", "spiky", 1024, 1024, 64),
        # a program whose timestamps live on the host: copies in, search, copies out
        _case("host_n1024_R1024_B64", "host", "range", "spiky", 1024, 1024, 64),
        # a server thread that may not allocate, deciding for a few mid-size jobs
        _case("noalloc_n100_R150_B4", "noalloc", "range", "lognormal", 100, 150, 4),
    ]


# most timestamps of a drawn case (n * R * B), and most instances
LIMITS = {"select_range": (1 << 27, 4096), "select_sum": (1 << 26, 4096), "predict": (1 << 26, 4096), "host": (1 << 26, 4096),
          "noalloc": (1 << 21, 64)}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choices(("select", "predict", "host", "noalloc"), (7, 1, 1, 1))[0]
    objective = "range" if entry == "predict" or rng.random() < 0.7 else "sum"
    total, batch = LIMITS[entry + "_" + objective if entry == "select" else entry]
    recipe = rng.choice(sorted(RECIPES))
    while True:
        n, R = _log_int(rng, 2, 4096), _log_int(rng, 4, 4096)
        if n * R <= total:
            break
    B = _log_int(rng, 1, max(1, min(batch, total // (n * R))))
    case = _case("", entry, objective, recipe, n, R, B, entry == "select" and rng.random() < 0.2)
    del case["name"]
    return case


def _worker_means(gen, recipe, B, n):
    """[B, n, 1] float64: mean iteration time of every worker."""
    r = RECIPES[recipe]
    if "second" in r:
        m = torch.full((B, n, 1), r["second"], dtype=torch.float64, device=gen.device)
        m[:, : n // 2] = r["mean"]
        return m
    m = r["mean"] * torch.exp(r["sigma"] * torch.randn((B, n, 1), generator=gen, dtype=torch.float64, device=gen.device))
    if "slow_share" in r:
        slow = math.ceil(r["slow_share"] * n - 1e-9)
        order = torch.rand((B, n), generator=gen, device=gen.device).argsort(dim=1)
        m[(order < slow)] *= r["slow_by"]
    return m


def _lengths(gen, recipe, means, R):
    """[B, n, R] int64: iteration lengths, at least one microsecond each."""
    r = RECIPES[recipe]
    shape = (means.shape[0], means.shape[1], R)
    d = torch.randn(shape, generator=gen, dtype=torch.float32, device=gen.device).mul_(r["jitter"]).add_(1.0)
    if "spike_share" in r:
        spikes = torch.rand(shape, generator=gen, dtype=torch.float32, device=gen.device) < r["spike_share"]
        d.mul_(spikes.to(torch.float32).mul_(r["spike_by"] - 1.0).add_(1.0))
    return (d * means.to(torch.float32)).round_().to(torch.int64).clamp_(min=1)


def _timestamps(gen, case):
    """[B, n, R] int64 end timestamps, a group of instances at a time."""
    B, n, R, r = case["B"], case["n"], case["R"], RECIPES[case["recipe"]]
    ts = torch.empty((B, n, R), dtype=torch.int64, device=gen.device)
    group = max(1, (1 << 24) // (n * R))
    for b in range(0, B, group):
        part = ts[b: b + group]
        torch.cumsum(_lengths(gen, case["recipe"], _worker_means(gen, case["recipe"], part.shape[0], n), R), dim=2, out=part)
        if "offset" in r:
            part += (torch.rand((part.shape[0], n, 1), generator=gen, dtype=torch.float64, device=gen.device) * r["offset"]).to(torch.int64)
    return ts


def prepare(case, seed):
    B, n, R = case["B"], case["n"], case["R"]
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    objective, entry = OBJECTIVES[case["objective"]], case["entry"]
    flags = zl.ZL_FLAG_CHECK_SORTED if case["checked"] else 0
    state = {"entry": entry, "objective": objective}
    where = {"device": "cpu", "pin_memory": True} if entry == "host" else {"device": dev}
    state["out"] = zl.Selection(torch.empty((B, n), dtype=torch.int32, **where), torch.empty(B, dtype=torch.int64, **where),
                                torch.empty(B, dtype=torch.int64, **where), torch.empty(B, dtype=torch.int32, **where))
    if entry == "predict":
        means = _worker_means(gen, case["recipe"], B, n)
        state["interval"] = _lengths(gen, case["recipe"], means, 1).reshape(B, n)
        state["last"] = (torch.rand((B, n), generator=gen, dtype=torch.float64, device=dev) * means[:, :, 0]).to(torch.int64)
        flags |= zl.ZL_FLAG_PREDICTOR
    else:
        ts = _timestamps(gen, case)
        if entry == "host":
            pinned = torch.empty((B, n, R), dtype=torch.int64, pin_memory=True)
            pinned.copy_(ts)
            ts = pinned
        state["ts"] = ts
    if entry != "noalloc":
        state["handle"] = zl.ZipLine(n, R, B, objective, dev.index, flags)
    return state


def run(state):
    entry, out = state["entry"], state["out"]
    if entry == "select":
        state["handle"].select_batched(state["ts"], out)
    elif entry == "predict":
        state["handle"].predict_select_batched(state["last"], state["interval"], out)
    elif entry == "host":
        state["handle"].select_batched_host(state["ts"], out)
    else:
        zl.zl_select_batched_noalloc(state["ts"], out, state["objective"])
    return {"idx": out.idx, "barrier": out.barrier, "wait": out.wait, "status": out.status}


def _examined_share(case):
    """Expected share of the timestamps that are not after the end of the first row to run out: later ones cannot
    belong to a complete selection, so the RANGE search may leave them unread."""
    r, n = RECIPES[case["recipe"]], case["n"]
    if "second" in r:
        return 1.0 if n < 2 else (n // 2 + (n - n // 2) * r["mean"] / r["second"]) / n
    rng = np.random.default_rng(1)
    draws = max(4, 4096 // n)
    m = np.exp(r["sigma"] * rng.standard_normal((draws, n)))
    if "slow_share" in r:
        m[:, : math.ceil(r["slow_share"] * n - 1e-9)] *= r["slow_by"]
    return float((m.min(axis=1, keepdims=True) / m).mean())


def work(case):
    B, n, R = case["B"], case["n"], case["R"]
    out = B * (4 * n + 20)
    if case["entry"] == "predict":
        return {"bytes": 16 * B * n + out, "flops": 0}
    share = 1.0 if case["objective"] == "sum" or case["checked"] else _examined_share(case)
    return {"bytes": int(8 * B * n * R * share) + out, "flops": 0}


def tolerance(case):
    return "exact"
