"""Timed workloads of the colour-index kernelization library.

Each case is one pass through the public entry points, as a program that uses
the library calls them:

* ``dense``    a dense 0/1 bit matrix in pinned host memory: load, kernelize
               to the fixpoint, fetch the kernel, free the handle;
* ``cascade``  a handle that is kept (the same graph kernelized again, for
               instance for another option): reset, kernelize, fetch;
* ``sparse``   an edge list in pinned host memory: load, kernelize, fetch the
               surviving edges, free;
* ``support``  a handle of an edge list that is kept, with the incremental
               support schedule: reset, kernelize, fetch the surviving edges;
* ``batch``    many handles reset, kernelized by one batch call, and fetched;
* ``noalloc``  one graph whose bit matrix and outputs stay in device memory,
               through the entry point that allocates nothing;
* ``mlp_forward`` / ``mlp_step``  the edge-scoring network: inference over
               feature rows, and one training step (gradient and Adam).

Graphs are random and legally coloured: k-partite with a planted k-clique, or
Chung-Lu with power-law degrees, Zipf colour classes and five planted cliques.
They are drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2212_00574_gb300 as kz

PARAMS = 64 * 16 + 64 + 64 * 64 + 64 + 64 + 1


def listed():
    return [
        # a latency-bound single graph (the smallest configured one, n = 300)
        {"name": "dense_small", "kind": "dense", "n": 300, "k": 10, "p": 0.7},
        # the ordinary dense graph: already a fixpoint, one certifying pass
        {"name": "dense_mid", "kind": "dense", "n": 4096, "k": 20, "p": 0.92},
        # the largest single graph, 437M edges, host copies included
        {"name": "dense_large", "kind": "dense", "n": 32768, "k": 24, "p": 0.85},
        # a sparser ragged graph in the cascade regime (several sweeps), plain sweeps
        {"name": "cascade_mid", "kind": "cascade", "n": 9001, "k": 17, "p": 0.112, "schedule": "plain"},
        # the largest cascade: a few tens of plain sweeps at the full size
        {"name": "cascade_large", "kind": "cascade", "n": 32768, "k": 24, "p": 0.07, "schedule": "plain"},
        # a cascade by re-check sweeps, the schedule made for it
        {"name": "cascade_support", "kind": "cascade", "n": 16384, "k": 24, "p": 0.1, "schedule": "support"},
        # the large sparse power-law graph given as an edge list
        {"name": "sparse_large", "kind": "sparse", "n": 200000, "k": 12, "degree": 60.0},
        # incremental support counts on a kept sparse handle, a ragged size
        {"name": "sparse_support", "kind": "support", "n": 100003, "k": 12, "degree": 60.0},
        # a batch of graphs of uneven size and colour count
        {"name": "batch_256", "kind": "batch", "count": 256, "n_hi": 4096, "batch": "concurrent"},
        # a device-resident graph in a process that must not allocate
        {"name": "noalloc_mid", "kind": "noalloc", "n": 1501, "k": 12, "p": 0.3},
        # scoring the edges of a frontier
        {"name": "mlp_forward_1m", "kind": "mlp_forward", "rows": 1000003},
        # one training step at the batch size the trainer uses
        {"name": "mlp_step_4096", "kind": "mlp_step", "rows": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "cascade", "cascade", "sparse", "support", "batch", "noalloc",
                       "mlp_forward", "mlp_step"])
    if kind == "dense":
        return {"kind": kind, "n": _log_int(rng, 48, 30000), "k": rng.randint(6, 32),
                "p": round(rng.uniform(0.3, 0.95), 3)}
    if kind == "cascade":
        n, k = _log_int(rng, 1000, 20000), rng.randint(8, 32)
        common = rng.uniform(3.0, 9.0)  # common neighbours an edge expects in a class
        return {"kind": kind, "n": n, "k": k, "p": round(min(0.6, math.sqrt(common * k / n)), 4),
                "schedule": rng.choice(["plain", "plain", "support"])}
    if kind in ("sparse", "support"):
        # graphs small enough for bitset rows beside the edge lists, and graphs beyond them
        n = _log_int(rng, 10000, 40000) if rng.random() < 0.4 else _log_int(rng, 80000, 200000)
        return {"kind": kind, "n": n, "k": rng.randint(8, 16),
                "degree": round(rng.uniform(20.0, 60.0), 1)}
    if kind == "batch":
        return {"kind": kind, "count": _log_int(rng, 16, 256), "n_hi": _log_int(rng, 512, 4096),
                "batch": rng.choice(["concurrent", "fused"])}
    if kind == "noalloc":
        return {"kind": kind, "n": _log_int(rng, 48, 4096), "k": rng.randint(6, 32),
                "p": round(rng.uniform(0.2, 0.95), 3)}
    if kind == "mlp_forward":
        return {"kind": kind, "rows": _log_int(rng, 100, 4000000)}
    return {"kind": kind, "rows": _log_int(rng, 64, 65536)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 17)
    return g


def _one_per_class(colour, k, gen, count=1):
    """count x k vertex ids, a different random vertex of each class per row
    (classes with fewer members leave their column at -1)."""
    n = colour.numel()
    perm = torch.randperm(n, generator=gen, device="cuda")
    order = torch.argsort(colour[perm], stable=True)
    sorted_ids = perm[order]
    sizes = torch.bincount(colour, minlength=k)
    first = torch.cumsum(sizes, 0) - sizes
    rows = []
    for i in range(count):
        ids = sorted_ids[torch.clamp(first + i, max=max(n - 1, 0))]
        rows.append(torch.where(sizes > i, ids, torch.full_like(ids, -1)))
    return torch.stack(rows)


def _clique_pairs(ids):
    ids, _ = torch.sort(ids[ids >= 0])
    iu = torch.triu_indices(ids.numel(), ids.numel(), 1, device="cuda")
    return ids[iu[0]], ids[iu[1]]


def _kpartite(n, k, p, seed, planted=True):
    """colour int32[n] and the upper-triangle bit matrix int64[n, ceil(n/64)], on the GPU."""
    gen = _generator(seed)
    colour = torch.randint(0, k, (n,), generator=gen, device="cuda", dtype=torch.int32)
    words = (n + 63) // 64
    padded = torch.full((64 * words,), -1, dtype=torch.int32, device="cuda")
    padded[:n] = colour
    column = torch.arange(64 * words, device="cuda", dtype=torch.int32)
    weight = torch.ones(64, dtype=torch.int64, device="cuda") << torch.arange(64, device="cuda")
    bits = torch.empty((n, words), dtype=torch.int64, device="cuda")
    step = max(1, (1 << 25) // (64 * words))
    if planted and n >= k:
        cu, cv = _clique_pairs(_one_per_class(colour, k, gen)[0])
    else:
        cu = cv = torch.empty(0, dtype=torch.int64, device="cuda")
    for a in range(0, n, step):
        b = min(n, a + step)
        r = torch.rand((b - a, 64 * words), generator=gen, device="cuda") < p
        r &= (padded >= 0) & (padded != colour[a:b, None]) & (column > column[a:b, None])
        here = (cu >= a) & (cu < b)
        r[cu[here] - a, cv[here]] = True
        bits[a:b] = (r.view(b - a, words, 64).to(torch.int64) * weight).sum(-1)
    return colour, bits


def _chung_lu(n, k, degree, seed):
    """colour int32[n] and canonical edges int32[m, 2], on the GPU."""
    gen = _generator(seed)
    rng = np.random.default_rng(seed * 7919 + 17)
    share = np.arange(1, k + 1, dtype=np.float64) ** -1.2
    share /= share.sum()
    colour = torch.from_numpy(rng.choice(k, size=n, p=share).astype(np.int32)).cuda()
    total = degree * n / (1.0 - float((share * share).sum()))
    w = (1.0 - rng.random(n)) ** (-1.0 / 1.3)
    for _ in range(8):
        w *= total / w.sum()
        w = np.minimum(w, math.sqrt(w.sum()))
    cum = torch.from_numpy(np.cumsum(w)).cuda()
    ends = torch.rand((2, int(w.sum() / 2)), generator=gen, device="cuda", dtype=torch.float64) * cum[-1]
    e = torch.searchsorted(cum, ends).clamp_(max=n - 1)
    e = e[:, colour[e[0]] != colour[e[1]]]
    lo, hi = torch.minimum(e[0], e[1]), torch.maximum(e[0], e[1])
    keys = [lo * n + hi]
    for ids in _one_per_class(colour, k, gen, count=5):
        u, v = _clique_pairs(ids)
        keys.append(u * n + v)
    key = torch.unique(torch.cat(keys))
    edges = torch.stack([key // n, key % n], dim=1).to(torch.int32)
    return colour, edges


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h.numpy()


def _bit_buffer(n):
    words = max((n + 63) // 64, 1)
    return torch.empty((n, words), dtype=torch.int64, pin_memory=True).numpy().view(np.uint64)


def _weights(seed):
    rng = np.random.default_rng(seed)
    parts = [rng.normal(0, math.sqrt(2 / 16), 64 * 16), rng.normal(0, 0.1, 64),
             rng.normal(0, math.sqrt(2 / 64), 64 * 64), rng.normal(0, 0.1, 64),
             rng.normal(0, math.sqrt(1 / 64), 64), rng.normal(0, 0.1, 1)]
    return np.concatenate(parts).astype(np.float32)


def _features(rows, seed):
    gen = _generator(seed)
    x = torch.rand((rows, 16), generator=gen, device="cuda")
    x[:, 2:4] *= -0.2  # the colour-cover slack is at most zero
    x[:, 6:8] *= -1.0  # and degrees only fall
    y = (torch.rand((rows,), generator=gen, device="cuda") < x[:, 15] * 0.5).to(torch.float32)
    return x.contiguous(), y


class _Model:
    def __init__(self, weights):
        self.h = kz.kz_model_create(weights)

    def __del__(self):
        kz.kz_model_free(self.h)


def _batch_specs(case, seed):
    """Sizes, colour counts and densities from the case alone, edges from the seed."""
    rng = np.random.default_rng(case["count"] * 7919 + case["n_hi"])
    for j in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(64), math.log(case["n_hi"])))))
        yield n, int(rng.integers(6, 33)), float(rng.uniform(0.3, 0.95)), j % 2 == 0, seed * 1000 + j


def prepare(case, seed):
    kz.use_torch_allocator()
    kind = case["kind"]
    s = {"case": case}
    if kind in ("dense", "cascade"):
        colour, bits = _kpartite(case["n"], case["k"], case["p"], seed)
        s["colour"], s["bits"] = _pinned(colour), _pinned(bits).view(np.uint64)
        s["alive"] = np.zeros(case["n"], np.uint8)
        s["out"] = _bit_buffer(case["n"])
        if kind == "cascade":
            s["graph"] = kz.KernelGraph(case["n"], case["k"], s["colour"], bits=s["bits"])
            s["options"] = kz.kz_default_options(schedule=case["schedule"])
    elif kind in ("sparse", "support"):
        colour, edges = _chung_lu(case["n"], case["k"], case["degree"], seed)
        s["colour"], s["edges"] = _pinned(colour), _pinned(edges)
        s["kept"], s["kept_rows"] = np.zeros((int(1.1 * case["degree"] * case["n"] / 2) + 1000, 2), np.int32), 0
        if kind == "support":
            s["graph"] = kz.KernelGraph(case["n"], case["k"], s["colour"], edges=s["edges"])
            s["options"] = kz.kz_default_options(schedule="support")
    elif kind == "batch":
        s["graphs"], rows, words = [], 0, 0
        for n, k, p, planted, gseed in _batch_specs(case, seed):
            colour, bits = _kpartite(n, k, p, gseed, planted)
            s["graphs"].append(kz.KernelGraph(n, k, colour.cpu().numpy(), bits=bits.cpu().numpy().view(np.uint64)))
            rows, words = rows + n, words + n * ((n + 63) // 64)
        s["alive"] = np.zeros(rows, np.uint8)
        s["out"] = torch.empty(words, dtype=torch.int64, pin_memory=True).numpy().view(np.uint64)
        s["options"] = kz.kz_default_options(batch=case["batch"])
    elif kind == "noalloc":
        s["colour"], s["bits"] = _kpartite(case["n"], case["k"], case["p"], seed)
        s["alive"] = torch.zeros(case["n"], dtype=torch.uint8, device="cuda")
        s["out"] = torch.zeros_like(s["bits"])
        s["counts"] = torch.zeros(4, dtype=torch.int64, device="cuda")
    else:
        s["model"] = _Model(_weights(seed))
        s["x"], s["y"] = _features(case["rows"], seed)
        s["logits"] = torch.empty(case["rows"], dtype=torch.float32, device="cuda")
        s["grad"] = torch.empty(PARAMS, dtype=torch.float32, device="cuda")
        s["loss"] = torch.empty(1, dtype=torch.float32, device="cuda")
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _keep_edges(s, edges):
    """The surviving edges in the caller's table (zero rows after the last one)."""
    m = len(edges)
    s["kept"][:m] = edges
    s["kept"][m:s["kept_rows"]] = 0
    s["kept_rows"] = m
    return s["kept"]


def _kernel(stats):
    return [stats["sweeps"], stats["passes"], stats["n_live"], stats["m_live"]]


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "dense":
        h = kz.kz_load_graph_dense(case["n"], case["k"], s["colour"], s["bits"])
        kz.kz_kernelize(h)
        _, _, stats = kz.kz_fetch_kernel_dense(h, case["n"], out_bits=s["out"], out_alive=s["alive"])
        kz.kz_free_graph(h)
        return {"alive": s["alive"], "bits": s["out"].view(np.int64), "stats": _kernel(stats),
                "edge_tests": stats["edge_tests"]}
    if kind == "cascade":
        g = s["graph"]
        kz.kz_reset(g.h)
        kz.kz_kernelize(g.h, s["options"])
        _, _, stats = kz.kz_fetch_kernel_dense(g.h, case["n"], out_bits=s["out"], out_alive=s["alive"])
        return {"alive": s["alive"], "bits": s["out"].view(np.int64), "stats": _kernel(stats)}
    if kind == "sparse":
        h = kz.kz_load_graph(case["n"], case["k"], s["colour"], s["edges"])
        kz.kz_kernelize(h)
        alive, edges, stats = kz.kz_fetch_kernel(h, case["n"])
        kz.kz_free_graph(h)
        return {"alive": alive, "edges": _keep_edges(s, edges), "stats": _kernel(stats)}
    if kind == "support":
        g = s["graph"]
        kz.kz_reset(g.h)
        kz.kz_kernelize(g.h, s["options"])
        alive, edges, stats = kz.kz_fetch_kernel(g.h, case["n"])
        return {"alive": alive, "edges": _keep_edges(s, edges), "stats": _kernel(stats)}
    if kind == "batch":
        for g in s["graphs"]:
            kz.kz_reset(g.h)
        kz.kz_kernelize_batch([g.h for g in s["graphs"]], s["options"])
        row = word = 0
        stats = []
        for g in s["graphs"]:
            w = (g.n + 63) // 64
            _, _, st = kz.kz_fetch_kernel_dense(g.h, g.n, out_bits=s["out"][word:word + g.n * w].reshape(g.n, w),
                                                out_alive=s["alive"][row:row + g.n])
            stats.append(_kernel(st) + [st["edge_tests"]])
            row, word = row + g.n, word + g.n * w
        return {"alive": s["alive"], "bits": s["out"].view(np.int64), "stats": np.array(stats, np.int64)}
    if kind == "noalloc":
        kz.kz_kernelize_dense_noalloc(case["n"], case["k"], s["colour"].data_ptr(), s["bits"].data_ptr(),
                                      s["bits"].shape[1], 0, s["alive"].data_ptr(), s["out"].data_ptr(),
                                      s["counts"].data_ptr())
        return {"alive": s["alive"], "bits": s["out"], "counts": s["counts"]}
    if kind == "mlp_forward":
        kz.kz_mlp_forward(s["model"].h, s["x"].data_ptr(), case["rows"], s["logits"].data_ptr())
        return s["logits"]
    kz.kz_mlp_grad(s["model"].h, s["x"].data_ptr(), s["y"].data_ptr(), case["rows"], s["grad"].data_ptr(),
                   s["loss"].data_ptr())
    kz.kz_mlp_adam(s["model"].h, s["grad"].data_ptr(), 3e-3)
    return {"grad": s["grad"], "loss": s["loss"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _dense_work(n, k, p):
    """The bit matrix read once and written once, the flags; one class test
    per expected edge and needed class."""
    edges = p * 0.5 * n * n * (k - 1) / k
    return 2.0 * n * ((n + 63) // 64) * 8 + 5.0 * n, edges * (k - 2)


def work(case):
    kind = case["kind"]
    if kind in ("dense", "cascade", "noalloc"):
        b, f = _dense_work(case["n"], case["k"], case["p"])
    elif kind in ("sparse", "support"):
        edges = case["degree"] * case["n"] / 2
        b, f = 8.0 * edges + 5.0 * case["n"], edges * (case["k"] - 2)
    elif kind == "batch":
        # means over the recipe: n log-uniform in [64, n_hi], k and p uniform
        span = math.log(case["n_hi"] / 64.0)
        n2 = (case["n_hi"] ** 2 - 64.0 ** 2) / (2 * span)
        b, f = case["count"] * n2 / 4, case["count"] * 0.625 * 0.5 * n2 * 17
    elif kind == "mlp_forward":
        b, f = 68.0 * case["rows"], 10368.0 * case["rows"]
    else:
        b, f = 68.0 * case["rows"] + 26.0 * PARAMS, 3 * 10368.0 * case["rows"]
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# computed numbers in 64 bits
# ---------------------------------------------------------------------------

def _layers(seed):
    w = torch.from_numpy(_weights(seed)).cuda().double()
    sizes = [64 * 16, 64, 64 * 64, 64, 64, 1]
    w1, b1, w2, b2, w3, b3 = torch.split(w, sizes)
    return w1.view(64, 16), b1, w2.view(64, 64), b2, w3, b3


def exact(case, seed):
    if case["kind"] not in ("mlp_forward", "mlp_step"):
        return None
    w1, b1, w2, b2, w3, b3 = _layers(seed)
    x, y = _features(case["rows"], seed)
    x, y = x.double(), y.double()
    if case["kind"] == "mlp_forward":
        out = []
        for c in torch.split(x, 1 << 18):
            h = torch.relu(torch.relu(c @ w1.T + b1) @ w2.T + b2)
            out.append(h @ w3 + b3)
        return torch.cat(out)
    z1 = x @ w1.T + b1
    h1 = torch.relu(z1)
    z2 = h1 @ w2.T + b2
    h2 = torch.relu(z2)
    logit = h2 @ w3 + b3
    loss = torch.nn.functional.binary_cross_entropy_with_logits(logit, y)
    d = (torch.sigmoid(logit) - y) / x.shape[0]
    dz2 = d[:, None] * w3 * (z2 > 0)
    dz1 = (dz2 @ w2) * (z1 > 0)
    grad = torch.cat([(dz1.T @ x).reshape(-1), dz1.sum(0), (dz2.T @ h1).reshape(-1), dz2.sum(0), h2.T @ d,
                      d.sum().reshape(1)])
    return {"grad": grad, "loss": loss.reshape(1)}
