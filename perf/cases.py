"""Performance cases of the range-retrieval library.

Each case is work that a user's program has the library do through its public
entry points: single lookups, batched range search at its operating points and
off them (ragged sizes, int8, heavy radii, fp32 and FP8 traversal, doubling),
the exhaustive ground truth, the server and the graph construction.

The points are a Gaussian mixture with Zipf weights and near-duplicate families
(random recursive trees), the queries 38% perturbed copies of points and 62%
fresh draws, and the radius the 40th percentile of exact 1-NN distances, so
that most queries match nothing and the match counts are heavy-tailed.  A
program builds its index once and searches it with many batches: the index (and
the server on it) is kept per index shape, made from a fixed seed, and the
batch of queries (for the construction case: the points) comes from the case's
seed.  Results come as CSR; the program stores their ids and distances in its
own buffers, kept from batch to batch with room for the largest one.
"""
from __future__ import annotations

import math
import weakref
from collections import OrderedDict

import numpy as np
import torch

import paper_2502_13245_gb300 as rr

DEV = "cuda:0"
INDEX_FIELDS = ("dtype", "metric", "n", "d", "R", "L", "centres", "cap", "relabel")

# index shapes: the 10^4-point parity workload, the 10^6-point one, the 10^7-point recipe at 2*10^6 points
# (vectors and rows 8x the L2 cache), fp32 unit vectors under inner product, and an odd int8 shape
C0 = dict(dtype="u8", metric="l2", n=10_000, d=128, R=32, L=64, centres=100, cap=500, relabel=False)
C1 = dict(dtype="u8", metric="l2", n=1_000_000, d=128, R=64, L=128, centres=1000, cap=5000, relabel=False)
C3P = dict(dtype="u8", metric="l2", n=2_000_000, d=256, R=64, L=48, centres=5000, cap=20_000, relabel=True)
C2 = dict(dtype="f32", metric="ip", n=1_000_000, d=200, R=64, L=128, centres=1000, cap=5000, relabel=False)
ODD = dict(dtype="i8", metric="l2", n=50_021, d=100, R=24, L=48, centres=223, cap=500, relabel=False)

SEARCH = dict(op="search", variant="greedy_es", beam=64, vl=20, esr=1.0, persistent=0, tile=0, precision=0, expand=1,
              spread="one", where="device")


def listed():
    return [
        # the smallest call: one query, no early stop, results into the caller's buffers
        dict(C0, name="noalloc_one", op="noalloc", nq=1, beam=64, variant="beam", vl=20, esr=1.0),
        # an interactive lookup: one host query against the 10^6-point index, host result
        dict(C1, **SEARCH | dict(variant="greedy", where="host"), name="lookup_one", nq=1),
        # a ragged batch on an odd int8 index, library defaults for the launch, host result
        dict(ODD, **SEARCH | dict(variant="greedy", beam=33, where="host"), name="ragged_i8", nq=777),
        # the 10^6-point workload at its operating point
        dict(C1, **SEARCH | dict(variant="greedy", beam=192, persistent=1, tile=4), name="batch_1m", nq=10_000),
        # the benchmark's form (AP >= 0.95) on the 10^7-point recipe: device queries and results
        dict(C3P, **SEARCH | dict(beam=96, vl=100, esr=2.0, persistent=1, tile=8), name="batch_2m", nq=20_000),
        # the serving mix's radii (r, 1.5r, 2r) in one batch of 2,048: the in-radius expansion dominates
        dict(C3P, **SEARCH | dict(beam=96, vl=100, esr=2.0, spread="mix"), name="heavy_2m", nq=2048),
        # fp32 vectors, exact traversal, at the operating point
        dict(C2, **SEARCH | dict(beam=8), name="fp32_1m", nq=10_000),
        # the same searches through the FP8 traversal copy
        dict(C2, **SEARCH | dict(beam=8, precision=rr.RR_PREC_FP8), name="fp8_1m", nq=10_000),
        # beam doubling instead of the greedy expansion
        dict(C1, **SEARCH | dict(variant="doubling", beam=16), name="doubling_1m", nq=2000),
        # exact ground truth of a query sample
        dict(C3P, op="brute", name="truth_2m", nq=1000),
        # single requests through the server: a burst of 256, radii mixed, host results
        dict(C1, op="serve", variant="greedy", beam=192, spread="mix", name="serve_1m", nq=256),
        # index construction
        dict(op="build", dtype="u8", metric="l2", n=100_000, d=128, R=32, L=64, centres=316, cap=500, relabel=False,
             name="build_100k"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_index(rng, n_hi):
    dtype = rng.choice(["u8", "u8", "u8", "i8", "f32"])
    n = _log(rng, 5_000, n_hi)
    d = rng.choice([_log(rng, 24, 256), 64, 96, 128, 200, 256])
    return dict(dtype=dtype, metric="ip" if dtype == "f32" and rng.random() < 0.7 else "l2", n=n, d=d,
                R=rng.choice([16, 24, 32, 48, 64, 64, rng.randint(16, 80)]), L=rng.choice([48, 64, 96]),
                centres=max(20, int(n ** 0.5)), cap=max(200, n // 200), relabel=rng.random() < 0.3)


def draw(rng):
    most = max(_gathered(c) for c in listed() if c["op"] == "search" and c["spread"] == "one")
    while True:
        kind = rng.random()
        if kind < 0.62:
            c = dict(_draw_index(rng, 2_000_000), **SEARCH)
            c.update(variant=rng.choice(["greedy", "greedy_es", "greedy_es", "beam", "beam_es", "doubling_es",
                                         "doubling_warm"]),
                     beam=_log(rng, 8, 256), nq=_log(rng, 1, 20_000), where=rng.choice(["device", "device", "host"]),
                     persistent=rng.choice([0, 1]), tile=rng.choice([0, 2, 4, 8]))
            if c["nq"] < 32:
                c["variant"] = c["variant"].replace("_es", "")  # an early stop can leave a tiny batch without results
            if c["variant"].endswith("_es") and c["metric"] == "l2":
                c["vl"], c["esr"] = rng.choice([(20, 1.0), (50, 1.5), (100, 2.0)])
            if c["dtype"] == "f32" and rng.random() < 0.5:
                c["precision"] = rng.choice([rr.RR_PREC_BF16, rr.RR_PREC_FP8])
            if c["variant"] in ("greedy", "beam", "greedy_es") and rng.random() < 0.15:
                c["expand"] = 2
            if c["dtype"] != "f32" and c["variant"].startswith("greedy") and rng.random() < 0.3:
                c["spread"], c["nq"] = "mix", min(c["nq"], 1024)
            if c["variant"].startswith("doubling"):
                c["nq"], c["beam"] = min(c["nq"], 1500), min(c["beam"], 32)
                if c["n"] > 1_000_000:
                    continue
            if _gathered(c) > most:
                continue
        elif kind < 0.74:
            c = dict(_draw_index(rng, 500_000), op="brute", nq=_log(rng, 1, 2000))
        elif kind < 0.84:
            c = dict(_draw_index(rng, 100_000), op="build")
            if c["dtype"] == "f32" or (c["L"] > 64 and c["n"] > 50_000):
                continue
        elif kind < 0.92:
            c = dict(_draw_index(rng, 1_000_000), op="noalloc", variant="beam", vl=20, esr=1.0,
                     beam=_log(rng, 8, 256), nq=_log(rng, 1, 2000))
            if c["nq"] >= 32 and rng.random() < 0.5:
                c["variant"] = "beam_es"
        else:
            c = dict(_draw_index(rng, 1_000_000), op="serve", variant="greedy", beam=_log(rng, 16, 128), spread="one",
                     nq=_log(rng, 1, 1000))
        return c


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _finish(c, v):
    if c["dtype"] == "f32":
        return (v / v.norm(dim=1, keepdim=True)).float()
    return v.round().clamp_(0, 255)


def _mixture(c, seed):
    """Centres, weights, and the spread of a fresh draw and of a near-duplicate."""
    g = _gen(seed)
    if c["dtype"] == "f32":
        mu = torch.randn(c["centres"], c["d"], device=DEV, generator=g)
        mu = mu / mu.norm(dim=1, keepdim=True)
        sigma, near = 0.06, 0.01
    else:
        mu = 40.0 + 175.0 * torch.rand(c["centres"], c["d"], device=DEV, generator=g)
        sigma, near = 12.0, 2.0
    w = 1.0 / torch.arange(1, c["centres"] + 1, device=DEV, dtype=torch.float32)
    return mu, w / w.sum(), sigma, near


def _stored(c, v):
    if c["dtype"] == "f32":
        return v.contiguous()
    return (v - 128).to(torch.int8) if c["dtype"] == "i8" else v.to(torch.uint8)


def _points(c, seed):
    """n x d float points: 80% mixture draws, 20% near-duplicate families (random recursive trees)."""
    mu, w, sigma, near = _mixture(c, seed)
    g = _gen(seed + 1)
    n, d = c["n"], c["d"]
    n_dup = n // 5
    n_base = n - n_dup
    X = torch.empty(n, d, device=DEV)
    for s in range(0, n_base, 1 << 19):
        e = min(n_base, s + (1 << 19))
        a = torch.multinomial(w, e - s, replacement=True, generator=g)
        X[s:e] = _finish(c, mu[a] + sigma * torch.randn(e - s, d, device=DEV, generator=g))
    rng = np.random.default_rng(seed)
    sizes = np.minimum(np.ceil(rng.pareto(1.0, n_dup) + 1.0), c["cap"]).astype(np.int64)
    ends = np.cumsum(sizes)
    nf = int(np.searchsorted(ends, n_dup)) + 1
    ends = np.minimum(ends[:nf], n_dup)
    first = np.concatenate([[0], ends[:-1]])
    fam = np.repeat(np.arange(nf), ends - first)
    k = np.arange(n_dup) - first[fam]                       # member number within its family
    par = np.floor(rng.random(n_dup) * (k + 1)).astype(np.int64)   # 0: the root, j: member j - 1
    roots = rng.integers(0, n_base, nf)
    src = torch.from_numpy(np.where(par == 0, roots[fam], n_base + first[fam] + par - 1)).to(DEV)
    done = torch.zeros(n, dtype=torch.bool, device=DEV)
    done[:n_base] = True
    left = torch.arange(n_dup, device=DEV)
    while left.numel():                                     # generation by generation
        ready = done[src[left]]
        m = left[ready]
        X[n_base + m] = _finish(c, X[src[m]] + near * torch.randn(m.numel(), d, device=DEV, generator=g))
        done[n_base + m] = True
        left = left[~ready]
    return X[torch.randperm(n, device=DEV, generator=g)]


def _queries(c, X, nq, seed):
    """38% perturbed copies of points, the rest fresh draws of the index's mixture; stored type."""
    mu, w, sigma, near = _mixture(c, 1000)
    g = _gen(seed)
    n_near = int(round(0.38 * nq)) if nq >= 8 else nq
    ids = torch.randint(0, X.shape[0], (n_near,), device=DEV, generator=g)
    x = X[ids].float() + (128.0 if c["dtype"] == "i8" else 0.0)
    q = [x + near * torch.randn(n_near, c["d"], device=DEV, generator=g)]
    if nq > n_near:
        a = torch.multinomial(w, nq - n_near, replacement=True, generator=g)
        q.append(mu[a] + sigma * torch.randn(nq - n_near, c["d"], device=DEV, generator=g))
    q = _finish(c, torch.cat(q))
    return _stored(c, q[torch.randperm(nq, device=DEV, generator=g)])


def _start(X):
    """The point nearest to the coordinate-wise mean."""
    best, at = math.inf, 0
    mean = sum(x.double().sum(0) for x in X.split(1 << 19)) / X.shape[0]
    for s, x in zip(range(0, X.shape[0], 1 << 19), X.split(1 << 19)):
        d, i = (x.double() - mean).square_().sum(1).min(0)
        if float(d) < best:
            best, at = float(d), s + int(i)
    return at


def _radius(c, X):
    """The 40th percentile of the 1-NN distances of 1,000 queries (integers up to d = 256 are exact here)."""
    Q = _queries(c, X, 1000, 77).float()
    best = torch.full((1000,), math.inf, device=DEV, dtype=torch.float64)
    for x in X.split(1 << 18):
        x = x.float()
        ip = (Q @ x.T).double()
        if c["metric"] == "l2":
            ip = x.double().square().sum(1)[None] + Q.double().square().sum(1)[:, None] - 2.0 * ip
        else:
            ip = -ip
        best = torch.minimum(best, ip.min(1).values)
    r = float(best.sort().values[400])
    return float(round(r)) if c["dtype"] != "f32" else round(r, 4)


def _adjacency(c, X, start):
    metric = rr.RR_IP if c["metric"] == "ip" else rr.RR_L2
    alpha, passes = (1.0, 1) if metric == rr.RR_IP else (1.2, 2)
    if c["dtype"] == "f32":                                 # the GPU builder takes 8-bit vectors
        X = (X * (127.0 / float(X.abs().max()))).round().to(torch.int8)
    return rr.rr_build_graph(X, c["R"], c["L"], alpha, passes=passes, seed=1, start=start, metric=metric)[0]


_kept = OrderedDict()


class _Kept:
    """What a program keeps for an index: the handle, and a server where it serves single requests."""

    def __init__(self, c):
        self.X = _stored(c, _points(c, 1000))
        self.start = _start(self.X)
        self.radius = _radius(c, self.X)
        self.adj = _adjacency(c, self.X, self.start)
        self.metric = rr.RR_IP if c["metric"] == "ip" else rr.RR_L2
        self.index = rr.Index.from_arrays(self.X, self.adj, self.start, metric=self.metric)
        if c["relabel"]:
            self.index.relabel()
        self.servers, self.room = {}, {}
        torch.cuda.empty_cache()

    def server(self, variant, beam):
        if (variant, beam) not in self.servers:
            self.servers[variant, beam] = self.index.serve(workers=2, variant=variant, beam=beam)
        return self.servers[variant, beam]

    def close(self):
        for s in self.servers.values():
            s.close()
        self.index.close()


def _index(c):
    rr.load_library()
    key = tuple(c[k] for k in INDEX_FIELDS)
    if key not in _kept:
        while len(_kept) >= 10:
            _kept.popitem(last=False)[1].close()
        _kept[key] = _Kept(c)
    _kept.move_to_end(key)
    return _kept[key]


def _params(c, radius):
    p = dict(beam=c["beam"], es_visit_limit=c.get("vl", 20), persistent=c.get("persistent", 0),
             tile_hint=c.get("tile", 0), precision=c.get("precision", 0), expand=c.get("expand", 1))
    if c.get("esr", 1.0) != 1.0:
        p.update(es_radius_mode=1, es_radius=radius * c["esr"])
    return p


def _radii(c, radius, seed):
    if c.get("spread", "one") == "one":
        return radius
    r = radius * np.random.default_rng(seed).choice([1.0, 1.5, 2.0], c["nq"])
    return np.floor(r)


def _room(c, k):
    """Entries of the program's result buffers: what earlier batches of this form needed, with headroom."""
    key = tuple(c.get(f) for f in ("op", "nq", "variant", "beam", "vl", "esr", "precision", "expand", "spread"))
    if key not in k.room:
        most = 0
        for seed in (1, 2, 3):
            Q = _queries(c, k.X, c["nq"], seed)
            if c["op"] == "brute":
                res = rr.rr_brute_force(k.index.h, Q, k.radius, result_on_device=True)
            else:
                res = rr.rr_range_search(k.index.h, Q, _radii(c, k.radius, seed), c["variant"],
                                         rr.rr_params_init(**_params(c, k.radius)), result_on_device=True)[1]
            most = max(most, res.total)
            rr.rr_result_free(res)
        mixed = c["n"] // 4 if c.get("spread") == "mix" else 0
        k.room[key] = min(c["nq"] * c["n"], 2 * most + 4 * c["cap"] + mixed + 4096)
    return k.room[key]


def _buffers(c, entries, device):
    ft = torch.float32 if c["dtype"] == "f32" else torch.int32
    return [torch.zeros(entries, dtype=torch.int32, device=device), torch.zeros(entries, dtype=ft, device=device)]


def _store(c, buf, ids, dists):
    """ids and dists into the program's buffers (grown where a batch has more than any before it)."""
    if len(ids) > buf[0].numel():
        buf[:] = _buffers(c, 2 * len(ids), buf[0].device)
    for b, x in zip(buf, (ids, dists)):
        b[:len(x)].copy_(x if isinstance(x, torch.Tensor) else torch.from_numpy(x))
    return buf


def prepare(case, seed):
    c = case
    s = {"case": c, "op": c["op"]}
    if c["op"] == "build":
        rr.load_library()
        s["X"] = _stored(c, _points(c, 2000 + seed))
        s["start"] = _start(s["X"])
        return s
    k = _index(c)
    Q = _queries(c, k.X, c["nq"], 3000 + seed)
    s.update(kept=k, index=k.index, radius=_radii(c, k.radius, seed), Q=Q)
    host = c["op"] == "serve" or (c["op"] == "search" and c["where"] == "host")
    if host:
        s["Q"] = Q.cpu().numpy()
    if c["op"] != "noalloc":
        s["buf"] = _buffers(c, _room(c, k), "cpu" if host else DEV)
    if c["op"] == "search":
        s["params"] = _params(c, k.radius)
        if c["where"] == "device":
            s["P"] = rr.rr_params_init(**s["params"])
    elif c["op"] == "serve":
        s["server"] = k.server(c["variant"], c["beam"])
    elif c["op"] == "noalloc":
        s["P"] = rr.rr_params_init(**_params(c, k.radius))
        ft = torch.float32 if c["dtype"] == "f32" else torch.int32
        s["out"] = (torch.empty(c["nq"], dtype=torch.int32, device=DEV),
                    torch.empty(c["nq"], c["beam"], dtype=torch.int32, device=DEV),
                    torch.empty(c["nq"], c["beam"], dtype=ft, device=DEV))
    return s


# ------------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------------

class _Owner:
    """A device result, freed when the last tensor that shows one of its arrays is gone."""

    def __init__(self, res):
        weakref.finalize(self, rr.rr_result_free, res)


class _Array:
    def __init__(self, owner, ptr, n, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": typestr, "data": (ptr, False), "version": 3}


def _device_csr(s, res):
    own, dt = _Owner(res), "<f4" if res.dist_dtype else "<i4"

    def view(ptr, n, typestr):
        if n == 0:
            return torch.empty(0, dtype={"<f4": torch.float32, "<i4": torch.int32}[typestr], device=DEV)
        return torch.as_tensor(_Array(own, ptr, n, typestr), device=DEV)

    buf = _store(s["case"], s["buf"], view(res.ids, res.total, "<i4"), view(res.dists, res.total, dt))
    return {"offsets": view(res.offsets, res.nq + 1, "<i8"), "ids": buf[0], "dists": buf[1],
            "flags": view(res.flags, res.nq, "|u1")}


def _host_csr(s, r):
    buf = _store(s["case"], s["buf"], r.ids.view(np.int32), r.dists)
    return {"offsets": r.offsets, "ids": buf[0], "dists": buf[1], "flags": r.flags}


def run(state):
    s, c = state, state["case"]
    if s["op"] == "search":
        if c["where"] == "host":
            return _host_csr(s, s["index"].range_search(s["Q"], s["radius"], c["variant"], **s["params"]))
        return _device_csr(s, rr.rr_range_search(s["index"].h, s["Q"], s["radius"], c["variant"], s["P"],
                                                 result_on_device=True)[1])
    if s["op"] == "noalloc":
        rr.rr_beam_search_noalloc(s["index"].h, s["Q"], s["radius"], c["variant"], s["P"], *s["out"])
        return {"counts": s["out"][0], "ids": s["out"][1], "dists": s["out"][2]}
    if s["op"] == "serve":
        first = int(s["server"].submit(s["Q"], s["radius"])[0])
        return _host_csr(s, s["server"].collect(first, c["nq"], timeout_ms=60_000))
    if s["op"] == "brute":
        return _device_csr(s, rr.rr_brute_force(s["index"].h, s["Q"], s["radius"], result_on_device=True))
    adj, _ = rr.rr_build_graph(s["X"], c["R"], c["L"], 1.2, passes=2, seed=1, start=s["start"], metric=rr.RR_L2)
    return adj


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------

def _row(c):
    return c["d"] * (4 if c["dtype"] == "f32" else 1)


def _visits(c):
    """Alg. 1 visits every point of its final beam; an early-stopped search (about half of the queries) its vl."""
    return 0.5 * (c["beam"] + c["vl"]) if c["variant"].endswith("_es") and c["vl"] < c["beam"] else c["beam"]


def _gathered(c):
    """Bytes of the adjacency rows visited and of the distinct vectors evaluated (about a third of a row's)."""
    row = {0: _row(c), 1: 2 * c["d"], 2: c["d"]}[c.get("precision", 0)]
    per = c["nq"] * (_visits(dict(vl=20, **c) if "vl" not in c else c) * (4 * c["R"] + c["R"] / 3 * row) + _row(c))
    return per


def work(case):
    c = case
    if c["op"] == "build":
        # every point: a beam search of L visits, and the pruning of its visits; both passes
        per = 2 * c["L"] * (4 * c["R"] + c["R"] / 3 * c["d"])
        return {"bytes": c["n"] * (per + c["d"] + 4 * c["R"]), "flops": c["n"] * 2 * c["L"] * c["R"] / 3 * 2 * c["d"]}
    if c["op"] == "brute":
        return {"bytes": (c["n"] + c["nq"]) * _row(c), "flops": 2.0 * c["n"] * c["nq"] * c["d"]}
    g = _gathered(c)
    if c.get("spread", "one") == "mix":
        # the in-radius expansion: results a third of the time in a ball that holds about 0.2% of the points
        hits = c["nq"] / 3 * 0.002 * c["n"]
        g += hits * (4 * c["R"] + _row(c) + 8)
    return {"bytes": g, "flops": 2.0 * g / (4 if c["dtype"] == "f32" else 1)}


# ------------------------------------------------------------------------------------------------
# the same results in 64 bits
# ------------------------------------------------------------------------------------------------

def _dist64(c, q, x):
    """Distances along the last axis of broadcast float64 operands."""
    return (q - x).square().sum(-1) if c["metric"] == "l2" else -(q * x).sum(-1)


def _csr64(c, s, q, ids, d):
    o = torch.argsort(ids, stable=True)
    q, ids, d = q[o], ids[o], d[o]
    o = torch.argsort(d, stable=True)
    q, ids, d = q[o], ids[o], d[o]
    o = torch.argsort(q, stable=True)
    offsets = torch.zeros(c["nq"] + 1, dtype=torch.int64, device=DEV)
    offsets[1:] = torch.bincount(q, minlength=c["nq"]).cumsum(0)
    m = s["buf"][0].numel()
    if len(d) > m:
        m = 2 * len(d)
    pad = (0, m - len(d))
    return {"offsets": offsets, "ids": torch.nn.functional.pad(ids[o], pad), "dists": torch.nn.functional.pad(d[o], pad),
            "flags": None}


def _brute64(c, s):
    X, Q, r = s["kept"].X, s["Q"].double(), s["radius"]
    qs, ids, ds = [], [], []
    step = max(1, (1 << 26) // c["nq"])
    for b in range(0, c["n"], step):
        x = X[b:b + step].double()
        d = Q @ x.T
        d = x.square().sum(1)[None] + Q.square().sum(1)[:, None] - 2.0 * d if c["metric"] == "l2" else -d
        q, i = (d <= r).nonzero(as_tuple=True)
        qs.append(q)
        ids.append(i + b)
        ds.append(d[q, i])
    return _csr64(c, s, torch.cat(qs), torch.cat(ids), torch.cat(ds))


def _search64(c, s):
    """Alg. 1 with Alg. 5 over the whole batch, then Alg. 2 from the queries whose beam filled."""
    k, nq, b, R, n = s["kept"], c["nq"], c["beam"], c["R"], c["n"]
    X, r = k.X.double(), k.radius
    Q = torch.as_tensor(s["Q"], device=DEV).double()
    adj = torch.from_numpy(k.adj.astype(np.int64)).to(DEV)
    esr = r * c["esr"] if c["esr"] != 1.0 else r
    ids = torch.full((nq, b), n, dtype=torch.int64, device=DEV)
    d = torch.full((nq, b), math.inf, dtype=torch.float64, device=DEV)
    vis = torch.ones((nq, b), dtype=torch.bool, device=DEV)
    ids[:, 0] = k.start
    d[:, 0] = _dist64(c, Q, X[k.start][None])
    vis[:, 0] = False
    nvis = torch.zeros(nq, dtype=torch.int64, device=DEV)
    live = torch.arange(nq, device=DEV)
    while live.numel():
        at = (~vis[live]).int().argmax(1)
        go = ~vis[live].gather(1, at[:, None])[:, 0]
        dp = d[live].gather(1, at[:, None])[:, 0]
        if c["variant"].endswith("_es"):
            go &= ~((d[live][:, 0] > r) & (nvis[live] >= c["vl"]) & (dp > esr))
        live, at = live[go], at[go]
        if not live.numel():
            break
        vis[live, at] = True
        nvis[live] += 1
        cand = adj[ids[live, at]]
        ok = cand < n
        ok &= ~(cand[:, :, None] == ids[live][:, None, :]).any(2)
        x = X[cand.clamp(max=n - 1)]
        dc = torch.where(ok, _dist64(c, Q[live][:, None], x), math.inf)
        del x
        D = torch.cat([d[live], dc], 1)
        I = torch.cat([ids[live], torch.where(ok, cand, n)], 1)
        V = torch.cat([vis[live], ~ok], 1)
        o = D.argsort(dim=1, stable=True)[:, :b]
        d[live], ids[live], vis[live] = D.gather(1, o), I.gather(1, o), V.gather(1, o)
    inr = (d <= r) & (ids < n)
    q, j = inr.nonzero(as_tuple=True)
    keys, dist = q * n + ids[q, j], d[q, j]
    front = keys[(inr.sum(1) == b)[q]] if c["variant"].startswith("greedy") else keys[:0]
    seen = front.sort().values
    while front.numel():
        nxt = []
        for f in front.split(1 << 18):
            nb = adj[f % n]
            nxt.append((torch.div(f, n, rounding_mode="floor")[:, None] * n + nb)[nb < n].unique())
        nxt = torch.cat(nxt).unique()
        p = torch.searchsorted(seen, nxt).clamp(max=seen.numel() - 1)
        nxt = nxt[seen[p] != nxt]
        seen = torch.cat([seen, nxt]).sort().values
        dn = torch.cat([_dist64(c, Q[torch.div(f, n, rounding_mode="floor")], X[f % n])
                        for f in nxt.split(1 << 18)]) if nxt.numel() else nxt.double()
        front = nxt[dn <= r]
        keys, dist = torch.cat([keys, front]), torch.cat([dist, dn[dn <= r]])
    return _csr64(c, s, torch.div(keys, n, rounding_mode="floor"), keys % n, dist)


def exact(case, seed):
    """Distances in 64 bits.  8-bit searches return whole numbers, which have to be equal; the low-precision
    traversals and doubling reach a set of points that has no 64-bit counterpart."""
    c = case
    if c["op"] == "brute" and c["n"] * c["nq"] <= 4e9:
        return _brute64(c, prepare(c, seed))
    if c["op"] == "search" and c["dtype"] == "f32" and not c["precision"] and c["expand"] == 1 \
            and not c["variant"].startswith("doubling") and c["nq"] * c["R"] * (c["d"] + c["beam"]) < 4e8:
        return _search64(c, prepare(c, seed))
    return None
