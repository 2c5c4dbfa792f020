"""The work a user of this library has it do, as cases to be measured.

Every case is one call sequence through the public binding
(``paper_2502_14446_gb300.momenti``) on a seeded synthetic series:

* ``search``   hash a series and search it (``hash_all`` + ``topk``);
* ``multi``    the same for a range of dimensionalities (``topk_multi``);
* ``anytime``  hash a series, advance the search a given number of
  repetitions and read the candidates found so far;
* ``exact``    the exact all-pairs search on an index the program holds;
* ``batch``    many series of uneven sizes in one call (``topk_batch``);
* ``verify``   distances of given pairs of windows on an index held;
* ``sort``     the allocation-free index sort of a column of hash keys.

Outputs are what the caller reads: motif positions, dimension sets and
distances (float64, as the library re-verifies them), the stopping point and
the miss bound of a search (the bound, and the candidates' distances of an
unfinished search, derive from the traversal's float32 distances and are
returned in that precision), distances of pairs, sorted orders.
"""
import ctypes as C
import math
import random

import numpy as np
import torch

from paper_2502_14446_gb300 import momenti as mom
from paper_2502_14446_gb300 import synth

# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

SEARCH = dict(kind="search", recipe="sensor", dtype="f32", precision="f16x2", L=200, k=10,
              delta=0.05, host=False, one_off=False, tensoring=False, motifs=5)


def listed():
    return [
        # a short recording searched once, from host memory, with a handle made for it
        # and closed after it (sizes of the smoke run): launches, round trips and set-up
        dict(SEARCH, name="search_one_off_n1500", recipe="walk", dtype="f64", host=True,
             one_off=True, D=3, n=1500, w=50, d=2, k=2, delta=0.1, L=100, motifs=2),
        # the plain small workload: float64 host data, a program that keeps its handle
        dict(SEARCH, name="search_f64_n5000", recipe="walk", dtype="f64", host=True, D=4, n=5000,
             w=100, d=2, k=5, delta=0.1, motifs=2),
        # the plain float32 workload, resident on the device: the headline search
        dict(SEARCH, name="search_f32_n100000", D=8, n=100000, w=300, d=3),
        # an odd-sized series as the batching workload holds them, hashed by the float32 form
        dict(SEARCH, name="search_fp32hash_n40001", recipe="walk", precision="fp32", D=11, n=40001,
             w=200, d=4, k=5, motifs=2),
        # the wide precision workload on its n = 200000 prefix: the largest call
        dict(SEARCH, name="search_wide_n200000", recipe="spikes", D=32, n=200000, w=500, d=8,
             delta=0.01, motifs=10),
        # tensored repetitions (L = 14^2), the memory-saving option
        dict(SEARCH, name="search_tensoring_n50000", tensoring=True, L=196, D=8, n=50000, w=300, d=3),
        # motifs of 2, 3 and 4 dimensions from one traversal
        dict(SEARCH, kind="multi", name="multi_d2to4_n20000", D=8, n=20000, w=100, d=2, d_high=4, k=5,
             motifs=4),
        # the large workload's shape (64 dims, long windows) on a prefix: hashing, then a look at
        # what the first repetitions found
        dict(SEARCH, kind="anytime", name="anytime_d64_n100000", D=64, n=100000, w=1000, d=16, L=8,
             delta=0.01, steps=12, motifs=20),
        # the exact search alone, on the scalability workload's shape
        dict(SEARCH, kind="exact", name="exact_n100000", recipe="walk", D=5, n=100000, w=300, d=2,
             k=1, L=4, motifs=1),
        # twelve recordings of uneven length and width in one call
        dict(kind="batch", name="batch_12_series", count=12, n_lo=2000, n_hi=40000, threads=8),
        # distances of a list of pairs, in float64
        dict(SEARCH, kind="verify", name="verify_f64_20000_pairs", D=8, n=100000, w=300, d=3, L=1,
             pairs=20000, fp64=True),
        # one column of hash keys sorted without allocation, at its size limit
        dict(kind="sort", name="sort_262144_keys", m=262144, K=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the same ranges: series of 500 to 100000 points, 1 to
    64 dimensions, windows of 20 to 1000 points, every option listed above."""
    kind = rng.choice(["search"] * 6 + ["multi", "anytime", "exact", "exact", "batch", "verify", "sort"])
    if kind == "sort":
        return dict(kind="sort", m=_log(rng, 500, 262144), K=rng.choice([3, 4, 6, 8, 8, 8]))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 16), n_lo=2000, n_hi=_log(rng, 4000, 30000),
                    threads=rng.choice([2, 4, 8]))
    D = _log(rng, 1, 64)
    wide = D > 16
    dtype = rng.choice(["f32", "f32", "f32", "f64"])
    # at most the work of the largest listed case; the float64, the several-d and the wide
    # searches (which may need every window's nearest neighbour first) cost more per pair of windows
    top = int(min(100000, math.sqrt((1.5e10 if wide and kind != "anytime" else 1e11) / D)))
    if dtype == "f64":
        top = min(top, 8000 if wide else 25000)
    if kind == "multi":
        top = min(top, 20000 if not wide else 10000)
    n = _log(rng, 500, top)
    k = rng.choice([1, 2, 3, 5, 10])
    # room for k motifs: 2 k windows more than w / 2 apart, wherever the first ones fall
    w = max(20, min(_log(rng, 20, 1000), n // (8 + 4 * k)))
    d = min(D, max(1, int(math.ceil(D / 3)) if not wide else int(math.ceil(D / 4))))
    c = dict(SEARCH, kind=kind, recipe=rng.choice(["walk", "sensor", "spikes"]), dtype=dtype, D=D, n=n,
             w=w, d=d, k=k, delta=rng.choice([0.01, 0.05, 0.1]),
             precision=rng.choice(["f16x2", "f16x2", "fp32"]), host=rng.random() < 0.5,
             motifs=rng.randint(1, max(1, min(10, n // (8 * w)))))
    if kind == "search":
        c["L"] = rng.choice([10, 50, 100, 200, 200])
        c["one_off"] = rng.random() < 0.25 and n <= 20000
        c["tensoring"] = rng.random() < 0.2
    elif kind == "multi":
        c["d"] = rng.randint(1, D)
        c["d_high"] = min(D, c["d"] + rng.randint(0, 2))
        c["L"] = rng.choice([50, 100, 200])
    elif kind == "anytime":
        c["L"] = rng.choice([8, 32, 100])
        c["steps"] = rng.randint(1, 2 * c["L"])
    elif kind == "verify":
        c["L"] = 1
        c["pairs"] = _log(rng, 10, 40000)
        c["fp64"] = rng.random() < 0.5
    else:
        c["L"] = rng.choice([1, 4])
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _series(c, seed):
    """The workloads' recipes: random walks (with sinusoids, noise and sparse
    spikes), and motifs planted in d dimensions."""
    g = np.random.Generator(np.random.Philox(int(seed) + 17))
    T = synth.random_walk(g, c["D"], c["n"])
    if c["recipe"] != "walk":
        T += synth.sinusoids(g, c["D"], c["n"]) + 0.1 * g.standard_normal(T.shape)
    if c["recipe"] == "spikes":
        T += synth.spikes(g, c["D"], c["n"], 1e-4, 5.0)
    synth.plant_motifs(g, T, c["w"], c["motifs"], c["d"], 0.05)
    return np.ascontiguousarray(T, dtype=np.float64 if c["dtype"] == "f64" else np.float32)


def _params(c, seed):
    return dict(w=c["w"], d=c["d"], k=c["k"], delta=c["delta"], L=c["L"], seed=int(seed) & 0x7FFFFFFF,
                precision=mom.PREC_FP32 if c["precision"] == "fp32" else mom.PREC_F16X2,
                flags=mom.FLAG_TENSORING if c["tensoring"] else 0)


def _batch(c, seed):
    return synth.batch_form(int(seed) + 17, count=c["count"], n_lo=c["n_lo"], n_hi=c["n_hi"])


def _pairs(c, seed):
    g = np.random.Generator(np.random.Philox(int(seed) + 18))
    return g.integers(0, c["n"] - c["w"] + 1, size=(c["pairs"], 2))


def _keys(c, seed):
    """Hash strings as the index holds them: each value a rounded normal
    within a signed byte (plus 128), zero bytes beyond K, and neighbouring
    windows often alike."""
    g = np.random.Generator(np.random.Philox(int(seed) + 19))
    v = np.cumsum(g.standard_normal((8, c["m"])) * 3.0, axis=1)
    v = np.mod(v + 400.0, 160.0) - 80.0 + g.standard_normal(v.shape) * 8.0
    v = np.clip(np.floor(v), -128, 127).astype(np.int64) + 128
    key = np.zeros(c["m"], dtype=np.uint64)
    for q in range(c["K"]):
        key |= v[q].astype(np.uint64) << np.uint64(56 - 8 * q)
    return key


def prepare(case, seed):
    c = dict(case)
    s = {"case": c}
    if c["kind"] == "sort":
        s["keys"] = torch.from_numpy(_keys(c, seed).view(np.int64)).cuda()
        s["order"] = torch.zeros(c["m"], dtype=torch.int32, device="cuda")
        s["lcp"] = torch.zeros(c["m"], dtype=torch.uint8, device="cuda")
        return s
    if c["kind"] == "batch":
        wls = _batch(c, seed)
        s["series"] = [wl.series for wl in wls]
        s["params"] = [dict(w=wl.w, d=wl.d, k=wl.k, delta=wl.delta) for wl in wls]
        return s
    T = _series(c, seed)
    s["series"] = T if c["host"] else torch.from_numpy(T).cuda()
    s["params"] = _params(c, seed)
    if not c["one_off"]:
        s["handle"] = mom.Momenti(**s["params"])
    if c["kind"] in ("exact", "verify"):
        s["handle"].hash_all(s["series"])
    if c["kind"] == "verify":
        s["pairs"] = _pairs(c, seed)
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def _motifs(ms, k, bound=False):
    """A list of at most k motifs as arrays of k (-1 and infinity where there
    are fewer)."""
    out = {"a": np.full(k, -1, dtype=np.int64), "b": np.full(k, -1, dtype=np.int64),
           "dims": np.zeros(k, dtype=np.uint64), "dist_d": np.full(k, np.inf),
           "dist_max": np.full(k, np.inf)}
    if bound:
        out["fail_bound"] = np.full(k, np.inf, dtype=np.float32)
    for q, m in enumerate(ms):
        out["a"][q], out["b"][q] = m["a"], m["b"]
        out["dims"][q] = sum(1 << f for f in m["dims"])
        out["dist_d"][q], out["dist_max"][q] = m["dist_d"], m["dist_max"]
        if bound:
            out["fail_bound"][q] = m["fail_bound"]
    return out


def _search(h, s):
    h.hash_all(s["series"])
    ms, st = h.topk()
    return dict(_motifs(ms, s["case"]["k"], bound=True), stop=np.array([st["stop_i"], st["stop_j"]]))


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "search":
        if c["one_off"]:
            with mom.Momenti(**state["params"]) as h:
                return _search(h, state)
        return _search(state["handle"], state)
    if kind == "exact":
        return _motifs(state["handle"].topk_exact(), c["k"])
    if kind == "multi":
        h = state["handle"]
        h.hash_all(state["series"])
        per_d, _ = h.topk_multi(c["d"], c["d_high"])
        return [dict(_motifs(ms, c["k"], bound=True), stop=np.array(stop)) for ms, stop in per_d.values()]
    if kind == "anytime":
        h = state["handle"]
        h.hash_all(state["series"])
        h.search_begin()
        h.search_step(c["steps"])
        now, cursor = h.search_current()
        out = _motifs(now[c["d"]], c["k"], bound=True)
        out["dist_d"] = out["dist_d"].astype(np.float32)
        out["dist_max"] = out["dist_max"].astype(np.float32)
        return dict(out, cursor=np.array(cursor, dtype=np.int64), r=float(h.info()["r"]))
    if kind == "batch":
        res = mom.topk_batch(state["params"], state["series"], threads=c["threads"])
        each = [_motifs(ms, 5, bound=True) for ms, _ in res]
        return {name: np.stack([m[name] for m in each]) for name in each[0]}
    if kind == "verify":
        per, dd, mask = state["handle"].verify(state["pairs"], fp64=c["fp64"])
        if not c["fp64"]:
            per, dd = per.astype(np.float32), dd.astype(np.float32)
        return {"per_dim": per, "dist_d": dd, "dims": mask}
    if kind == "sort":
        rc = mom.lib.momenti_index_sort_noalloc(
            C.c_void_p(state["keys"].data_ptr()), c["m"], c["K"], C.c_void_p(state["order"].data_ptr()),
            C.c_void_p(state["lcp"].data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != mom.OK:
            raise mom.MomentiError(rc, "momenti_index_sort_noalloc")
        return {"order": state["order"], "lcp": state["lcp"]}
    raise ValueError(kind)


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _search_work(D, n, w, L, K, size, exact):
    M = n - w + 1
    # projections of every window on K L vectors per dimension, and the
    # sliding products (two FMA) and the threshold test (two FMA) of every
    # pair of windows and dimension where the search ends in the exact path
    # (as these do)
    flops = 2.0 * w * K * L * D * M + (8.0 * D * 0.5 * M * M if exact else 0.0)
    return {"bytes": float(size * D * n), "flops": flops}


def work(case):
    c = case
    if c["kind"] == "sort":
        return {"bytes": float(c["m"] * (8 + 4 + 1)), "flops": 0.0}
    if c["kind"] == "batch":
        # series lengths are drawn: their logarithmic mean, ten dimensions
        n = (c["n_hi"] - c["n_lo"]) / math.log(c["n_hi"] / c["n_lo"])
        one = _search_work(10, int(n), 100, 200, 8, 4, True)
        return {"bytes": one["bytes"] * c["count"], "flops": one["flops"] * c["count"]}
    size = 8 if c["dtype"] == "f64" else 4
    M = c["n"] - c["w"] + 1
    if c["kind"] == "verify":
        return {"bytes": float(min(size * c["D"] * c["n"], 2 * size * c["D"] * c["w"] * c["pairs"])
                               + 8 * c["pairs"] * (2 + c["D"] + 2)),
                "flops": 7.0 * c["pairs"] * c["D"] * c["w"]}
    if c["kind"] == "exact":
        return {"bytes": float(size * c["D"] * c["n"]), "flops": 8.0 * c["D"] * 0.5 * M * M}
    if c["tensoring"]:
        # 2 sqrt(L) half functions of K / 2 values
        return _search_work(c["D"], c["n"], c["w"], 2 * math.isqrt(c["L"]), 4, size, True)
    return _search_work(c["D"], c["n"], c["w"], c["L"], 8, size, c["kind"] != "anytime")


# --------------------------------------------------------------------------
# the results in 64 bits
# --------------------------------------------------------------------------

def _windows(T, w):
    """z-normalised windows of one dimension (population sigma; a flat
    window is the zero vector), (M, w) float64 on the device."""
    x = torch.from_numpy(np.asarray(T, dtype=np.float64)).cuda().unfold(0, w, 1)
    mu = x.mean(dim=1, keepdim=True)
    z = x - mu
    sd = z.square().mean(dim=1, keepdim=True).sqrt()
    return torch.where(sd <= 1e-8 * (1.0 + mu.abs()), torch.zeros_like(z), z / sd)


def _pair_dists(Z, a, b):
    return torch.stack([(z[a] - z[b]).square().sum(dim=-1).sqrt() for z in Z], dim=-1)


def _exact_topk(T, w, ds, k):
    """The exact top-k motifs of every d of ds: greedy in ascending distance
    under the exclusion zone w / 2."""
    D, M, eps = T.shape[0], T.shape[1] - w + 1, w // 2
    Z = [_windows(T[f], w) for f in range(D)]
    full = {d: torch.empty((M, M), dtype=torch.float64, device="cuda") for d in ds}
    col = torch.arange(M, device="cuda")
    step = max(1, min(M, int(5e8 // (D * M))))
    for r0 in range(0, M, step):
        r1 = min(M, r0 + step)
        sq = torch.stack([z[r0:r1].square().sum(1)[:, None] + z.square().sum(1)[None, :]
                          - 2.0 * (z[r0:r1] @ z.T) for z in Z])
        best = sq.clamp_(min=0.0).sqrt_().sort(dim=0).values.cumsum(dim=0)
        trivial = col[None, :] - torch.arange(r0, r1, device="cuda")[:, None] <= eps
        for d in ds:
            full[d][r0:r1] = best[d - 1].masked_fill(trivial, math.inf)
    out = {}
    for d in ds:
        m, ms = full[d], []
        for _ in range(k):
            q = int(m.argmin())
            a, b = q // M, q % M
            if not math.isfinite(float(m[a, b])):
                break
            per = _pair_dists(Z, a, b)
            val, dim = per.sort(stable=True)
            ms.append({"a": a, "b": b, "dist_d": float(val[:d].sum()), "dist_max": float(val[d - 1]),
                       "dims": tuple(int(f) for f in dim[:d])})
            for x in (a, b):
                lo, hi = max(0, x - eps), x + eps + 1
                m[lo:hi] = math.inf
                m[:, lo:hi] = math.inf
        ms.sort(key=lambda t: (t["dist_d"], t["a"], t["b"]))
        out[d] = _motifs(ms, k)
    return out


def exact(case, seed):
    c = case
    if c["kind"] == "sort":
        key = _keys(c, seed)
        order = np.argsort(key, kind="stable")
        s = key[order]
        x = s[1:] ^ s[:-1]
        lcp = np.zeros(c["m"], dtype=np.uint8)
        same = np.full(c["m"] - 1, c["K"], dtype=np.uint8)
        for q in range(c["K"] - 1, -1, -1):
            same[(x >> np.uint64(56 - 8 * q)) & np.uint64(255) != 0] = q
        lcp[1:] = same
        return {"order": order.astype(np.int32), "lcp": lcp}
    if c["kind"] in ("batch", "anytime"):
        return None
    T = _series(c, seed)
    if c["kind"] == "verify":
        p = torch.from_numpy(_pairs(c, seed)).cuda()
        per = torch.empty((c["pairs"], c["D"]), dtype=torch.float64, device="cuda")
        for f in range(c["D"]):
            per[:, f] = _pair_dists([_windows(T[f], c["w"])], p[:, 0], p[:, 1])[:, 0]
        val, dim = per.sort(dim=1, stable=True)
        mask = np.zeros(c["pairs"], dtype=np.uint64)
        for q in range(c["d"]):
            mask |= np.uint64(1) << dim[:, q].cpu().numpy().astype(np.uint64)
        return {"per_dim": per.cpu().numpy(), "dist_d": val[:, :c["d"]].sum(dim=1).cpu().numpy(), "dims": mask}
    M = c["n"] - c["w"] + 1
    if M > 20000 or float(M) * M * c["D"] * c["w"] > 1.5e12:
        return None
    if c["kind"] == "multi":
        ds = list(range(c["d"], c["d_high"] + 1))
        res = _exact_topk(T, c["w"], ds, c["k"])
        return [dict(res[d], fail_bound=None, stop=None) for d in ds]
    res = _exact_topk(T, c["w"], [c["d"]], c["k"])[c["d"]]
    return res if c["kind"] == "exact" else dict(res, fail_bound=None, stop=None)
