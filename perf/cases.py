"""Timed workloads of the U-HNSW library, through its public entry points.

Every case is a call that a user of the library makes: a search (plain,
persistent, CUDA-graph replay, host buffers, the batching server), the
verification of given candidate lists, the exhaustive search, and the
construction of a graph.  A search case keeps one loaded index per data set
and storage type, as a program that serves queries does (the base vectors and
graphs come from a fixed stream, built once per process); the queries, their
p, k and ef come from the seed.  The build case's base vectors come from the
seed, its node levels from a fixed stream.

Data sets (the recipes of paper_2605_02030_gb300/inputs.py, drawn on the GPU):
  sift     integer features 0..255 around n_clusters centres, SIFT-shaped
  mixture  Gaussian mixture, unit noise around N(0, 4I) centres
  gist     values in [0, 1], a Beta mixture of 100 clusters, GIST-shaped
  unit     N(0, I) rows scaled to unit L2 norm
"""
import functools
import math

import numpy as np
import torch

from paper_2605_02030_gb300 import inputs as I
from paper_2605_02030_gb300 import uhnsw as U

DEV = "cuda"
CLUSTERS = {"sift": 1000, "mixture": 16, "gist": 100}
P_GRID = [0.5 + 0.1 * i for i in range(16)]
BYTES = {"f32": 4, "f16": 2, "bf16": 2}


def listed():
    sift = dict(data="sift", n=1_000_000, d=128, M=32, efc=200)
    unit = dict(data="unit", n=1_000_000, d=96, M=32, efc=200)
    return [
        # one user request answered by itself: latency alone
        dict(name="one_query", do="search", **sift, dtype="f16", graphs="u", form="plain", nq=1,
             k=10, ef=64, width=1, p="uniform"),
        # the small configuration: 100 queries of a 10,000 x 32 FP32 index
        dict(name="mixture_100", do="search", data="mixture", n=10_000, d=32, M=16, efc=100,
             dtype="f32", graphs="u", form="plain", nq=100, k=10, ef=64, width=1, p="uniform"),
        # the precision form in batches, at the operating point of the benchmark
        dict(name="sift_batched_f16", do="search", **sift, dtype="f16", graphs="u", form="graph",
             nq=10_000, k=10, ef=52, width=2, p="uniform"),
        # the plain form: FP32 rows, HNSW's own order, one launch per batch
        dict(name="sift_plain_f32", do="search", **sift, dtype="f32", graphs="u", form="plain",
             nq=10_000, k=10, ef=64, width=1, p="grid"),
        # a service that holds its queries in host memory
        dict(name="sift_host_1000", do="search", **sift, dtype="f16", graphs="u", form="host",
             nq=1_000, k=10, ef=64, width=2, p="uniform"),
        # the batched form: wide BF16 rows, every query with its own p, k and ef
        dict(name="gist_mixed_bf16", do="search", data="gist", n=100_000, d=960, M=32, efc=200,
             dtype="bf16", graphs="u", form="persistent", nq=10_000, k=0, ef=0, width=1,
             p="uniform"),
        # a batch as the serving form launches it, at the largest beam
        dict(name="unit_ef512", do="search", **unit, dtype="f16", graphs="u", form="plain",
             nq=1_000, k=0, ef=512, width=1, p="uniform"),
        # requests that reach the server at once: continuous batching, several batches in flight
        dict(name="unit_serve_burst", do="search", **unit, dtype="f16", graphs="u", form="serve",
             nq=2_048, k=0, ef=512, width=1, p="uniform"),
        # U-HNSW-E: graphs under L0.5 and L1, p below 0.7
        dict(name="sift_e_f16", do="search", **sift, dtype="f16", graphs="e", form="persistent",
             nq=10_000, k=10, ef=72, width=2, p="low"),
        # re-ranking alone, at the paper's t = 300 and K = 50
        dict(name="verify_300", do="verify", data="sift", n=1_000_000, d=128, nq=5_003, t=300, k=50,
             mode="exact", p="uniform"),
        # exhaustive answers for recall
        dict(name="exact_1001", do="exact", data="sift", n=1_000_000, d=128, nq=1_001, k=10,
             p="uniform"),
        # construction of one graph on the GPU
        dict(name="build_gpu", do="build", data="sift", n=50_000, d=128, metric=1, M=32, efc=200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    if u < 0.6:
        which = rng.choice(["sift", "sift", "mixture", "gist", "unit"])
        if which == "sift":
            c = dict(data="sift", n=1_000_000, d=128, M=32, efc=200)
            c["dtype"] = rng.choice(["f16", "f16", "f32", "bf16"])
        elif which == "mixture":
            c = dict(data="mixture", n=_log(rng, 2_000, 50_000), d=rng.randint(8, 200),
                     M=rng.choice([8, 16, 24]), efc=100, dtype=rng.choice(["f32", "f16", "bf16"]))
        elif which == "gist":
            c = dict(data="gist", n=_log(rng, 5_000, 40_000), d=rng.choice([960, 500, 1023]), M=16,
                     efc=100, dtype=rng.choice(["bf16", "f16", "f32"]))
        else:
            c = dict(data="unit", n=_log(rng, 20_000, 200_000), d=96, M=32, efc=100,
                     dtype=rng.choice(["f16", "f16", "f32"]))
        c.update(do="search", graphs=rng.choice(["u", "u", "u", "e"]),
                 form=rng.choice(["plain", "plain", "persistent", "graph", "host"]),
                 nq=_log(rng, 1, 10_000), width=rng.choice([1, 1, 2, 3]))
        c["p"] = "low" if c["graphs"] == "e" else rng.choice(["uniform", "uniform", "grid"])
        c["k"] = rng.choice([0, _log(rng, 1, 100)])
        c["ef"] = rng.choice([0, max(c["k"], _log(rng, 10, 512))])
        most = work(listed()[5])["bytes"]
        while c["nq"] > 1 and work(c)["bytes"] > most:
            c["nq"] = max(1, c["nq"] // 2)
        return c
    if u < 0.75:
        data, n, d = rng.choice([("sift", 1_000_000, 128), ("mixture", 40_000, rng.randint(8, 300)),
                                 ("gist", 60_000, 960)])
        t = _log(rng, 10, 512)
        nq = _log(rng, 1, 10_000)
        return dict(do="verify", data=data, n=n, d=d, nq=max(1, min(nq, 200_000_000 // (t * d))), t=t,
                    k=min(t, _log(rng, 1, 100)), mode=rng.choice(["exact", "paper"]),
                    p=rng.choice(["uniform", "grid", "low"]))
    if u < 0.9:
        data, n, d = rng.choice([("sift", 1_000_000, 128), ("mixture", _log(rng, 1_000, 300_000), 32),
                                 ("mixture", _log(rng, 1_000, 100_000), rng.randint(8, 200)),
                                 ("gist", 50_000, 960)])
        nq = max(1, min(_log(rng, 1, 4_000), 128_000_000_000 // (n * d)))
        return dict(do="exact", data=data, n=n, d=d, nq=nq, k=_log(rng, 1, 256),
                    p=rng.choice(["uniform", "grid", "low"]))
    data, d = rng.choice([("sift", 128), ("mixture", rng.randint(8, 150)), ("unit", 96)])
    return dict(do="build", data=data, n=_log(rng, 3_000, 50_000), d=d, metric=rng.choice([1, 2, 2, 3]),
                M=rng.choice([8, 16, 32]), efc=rng.choice([64, 100, 200]))


# ---------------------------------------------------------------- inputs (torch alone)
def _gen(*seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(np.random.SeedSequence([int(s) for s in seed]).generate_state(1, np.uint64)[0] >> 1))
    return g


@functools.lru_cache(maxsize=None)
def _centres(data, d):
    g = _gen(1, len(data), d)
    c = CLUSTERS[data]
    if data == "mixture":
        return torch.randn((c, d), generator=g, device=DEV) * 2.0
    if data == "sift":
        e = -30.0 * torch.log1p(-torch.rand((c, d), generator=g, device=DEV))
        return e.clamp_(0, 255)
    with torch.random.fork_rng(devices=[torch.cuda.current_device()]):
        torch.manual_seed(17 + d)
        two, five = (torch.full((c, d), v, device=DEV) for v in (2.0, 5.0))
        return torch.distributions.Beta(two, five).sample()


def _points(data, d, cluster, g, n):
    """n rows, row i around centre cluster[i] (no centre for unit rows)."""
    if data == "unit":
        x = torch.randn((n, d), generator=g, device=DEV)
        return x / x.norm(dim=1, keepdim=True)
    c = _centres(data, d)[cluster]
    if data == "mixture":
        return c + torch.randn((n, d), generator=g, device=DEV)
    if data == "sift":
        return (c + 20.0 * torch.randn((n, d), generator=g, device=DEV)).clamp_(0, 255).round_()
    c = c.clamp_(1e-3, 1 - 1e-3)
    with torch.random.fork_rng(devices=[torch.cuda.current_device()]):
        torch.manual_seed(g.initial_seed() % (1 << 62))
        return torch.distributions.Beta(20.0 * c, 20.0 * (1.0 - c)).sample()


def _base_dev(data, n, d, seed=0):
    """Base rows on the GPU; row i lies around centre i % n_clusters."""
    rows = torch.arange(n, device=DEV) % CLUSTERS.get(data, 1)
    return _points(data, d, rows, _gen(2, seed, n, d), n).contiguous()


@functools.lru_cache(maxsize=3)
def _base(data, n, d):
    return _base_dev(data, n, d).cpu().numpy()


def _queries(data, d, nq, pmode, seed):
    """(q [nq, d], cluster [nq], p [nq]) on the GPU."""
    g = _gen(3, seed, nq, d)
    cl = torch.randint(0, CLUSTERS.get(data, 1), (nq,), generator=g, device=DEV)
    q = _points(data, d, cl, g, nq).contiguous()
    u = torch.rand((nq,), generator=g, device=DEV)
    if pmode == "grid":
        p = torch.tensor(P_GRID, device=DEV)[(u * len(P_GRID)).long().clamp_(max=len(P_GRID) - 1)]
    else:
        lo, hi = (0.2, 0.7) if pmode == "low" else (0.5, 2.0)
        p = hi - (hi - lo) * u
    return q, cl, p.float().contiguous()


def _candidates(base, q, cl, n, t, clusters):
    """The t rows of each query's own cluster that are nearest under L1, ascending."""
    per = n // clusters
    out = torch.empty((q.shape[0], t), dtype=torch.int32, device=DEV)
    step = max(1, (1 << 29) // (per * q.shape[1] * 4))
    member = torch.arange(per, device=DEV) * clusters
    for s in range(0, q.shape[0], step):
        ids = member[None, :] + cl[s:s + step, None]
        dist = (base[ids.reshape(-1)].view(ids.shape[0], per, -1) - q[s:s + step, None]).abs_().sum(-1)
        order = torch.sort(dist, dim=1, stable=True).indices[:, :t]
        out[s:s + step] = torch.gather(ids, 1, order).int()
    return out.contiguous()


# ---------------------------------------------------------------- the index a program keeps
@functools.lru_cache(maxsize=6)
def _graph(data, n, d, metric, M, efc):
    lv = I.hnsw_levels(n, M, 11 + metric)
    return U.build_graph(_base(data, n, d), metric, M, efc, lv, device="gpu")


@functools.lru_cache(maxsize=8)
def _index(data, n, d, M, efc, dtype, graphs):
    metrics = U.U_HNSW_E if graphs == "e" else U.U_HNSW
    g = [_graph(data, n, d, m, M, efc) for m in metrics]
    return U.Index(_base(data, n, d), g[0], g[1], traverse_dtype=dtype, metrics=metrics)


@functools.lru_cache(maxsize=4)
def _bare_index(data, n, d):
    """An index for calls that use the rows alone: one cheap graph."""
    nbr = np.arange(1, n + 1, dtype=np.int32) % n
    level = {"nodes": np.arange(n, dtype=np.int32), "offsets": np.arange(n + 1, dtype=np.int64), "nbrs": nbr}
    chain = {"num_levels": 1, "entry_point": 0, "max_degree0": 1, "max_degree": 1, "n": n,
             "levels": [level]}
    return U.Index(_base(data, n, d), chain, None)


# ---------------------------------------------------------------- the cases
def prepare(case, seed):
    do, data, n, d = case["do"], case["data"], case["n"], case["d"]
    s = {"case": case}
    if do == "build":
        s["base"] = _base_dev(data, n, d, seed + 1).cpu().numpy()
        s["levels"] = I.hnsw_levels(n, case["M"], 5)
        return s
    q, cl, p = _queries(data, d, case["nq"], case["p"], seed)
    s.update(q=q, p=p)
    if do == "verify":
        s["cand"] = _candidates(_base_dev(data, n, d), q, cl, n, case["t"], CLUSTERS[data])
        s["index"] = _bare_index(data, n, d)
        return s
    if do == "exact":
        s["index"] = _bare_index(data, n, d)
        return s
    s["index"] = _index(data, n, d, case["M"], case["efc"], case["dtype"], case["graphs"])
    nq, k, ef = case["nq"], case["k"], case["ef"]
    g = _gen(4, seed, nq)
    # the k and ef of each query where the case does not give one for all
    ks = [1, 10, 100] if data == "gist" else [10, 50]
    k_q = torch.tensor(ks, dtype=torch.int32, device=DEV)[
        torch.randint(0, len(ks), (nq,), generator=g, device=DEV)]
    efs = [32, 64, 128, 256, 512]
    ef_q = torch.tensor(efs, dtype=torch.int32, device=DEV)[
        torch.randint(0, len(efs), (nq,), generator=g, device=DEV)]
    ef_q = torch.maximum(ef_q, k_q if not k else torch.full_like(k_q, k))
    k_max = k or max(ks)
    s["k"] = k or k_q.contiguous()
    s["ef"] = ef_q.contiguous() if not ef else ef if k else max(ef, k_max)
    s["opts"] = dict(k_max=k_max, width=case["width"],
                     persistent=case["form"] in ("persistent", "graph", "host"),
                     cutoff=0.6 if case["graphs"] == "e" else 0.0)
    if not ef:
        s["opts"]["ef_max"] = 512
    if case["form"] == "graph":
        s["opts"].update(use_graph=True, out=(torch.empty((nq, k_max), dtype=torch.int64, device=DEV),
                                              torch.empty((nq, k_max), device=DEV)))
    elif case["form"] == "host":
        def pin(t):
            return t.cpu().pin_memory().numpy() if torch.is_tensor(t) else t
        s.update(q=pin(q), p=pin(p), k=pin(s["k"]), ef=pin(s["ef"]))
    elif case["form"] == "serve":
        s.update(q=q.cpu().numpy(), p=p.cpu().numpy())
        s["k"], s["ef"] = (v.cpu().numpy() if torch.is_tensor(v) else v for v in (s["k"], s["ef"]))
        s["arrival"] = np.zeros(nq)
        s["server"] = U.Server(s["index"], k_max=k_max, ef_max=512, width=case["width"],
                               cutoff=s["opts"]["cutoff"])
    return s


def _whole(g, l):
    """One level of a built graph; its links, whose number depends on the rows, filled up to the cap."""
    lv = g["levels"][l]
    links = np.full(len(lv["nodes"]) * g["max_degree0" if l == 0 else "max_degree"], -1, np.int32)
    links[:len(lv["nbrs"])] = lv["nbrs"]
    return {"nodes": lv["nodes"], "offsets": lv["offsets"], "links": links}


def run(s):
    case = s["case"]
    if case["do"] == "build":
        g = U.build_graph(s["base"], case["metric"], case["M"], case["efc"], s["levels"], device="gpu")
        return {"entry": g["entry_point"], "levels": [_whole(g, l) for l in range(g["num_levels"])]}
    if case["do"] == "verify":
        ids, dist, _ = s["index"].verify(s["q"], s["p"], s["cand"], case["k"], mode=case["mode"])
        return ids, dist
    if case["do"] == "exact":
        return s["index"].exact(s["q"], s["p"], case["k"])
    if case["form"] == "serve":
        ids, dist, _ = s["server"].replay(s["q"], s["p"], s["k"], s["ef"], s["arrival"])
        return ids, dist
    if case["form"] == "host":
        return s["index"].search_host(s["q"], s["p"], s["k"], s["ef"], **s["opts"])
    ids, dist, _ = s["index"].search(s["q"], s["p"], s["k"], s["ef"], **s["opts"])
    return ids, dist


def work(case):
    """Bytes and operations of one pass.  A search of beam ef expands about ef
    nodes (2M links each) and evaluates about M rows per expansion, and
    verifies its ef candidates on their FP32 rows; an insertion is such a
    search at efConstruction."""
    n, d, do = case["n"], case["d"], case["do"]
    if do == "exact":
        nq = case["nq"]
        return {"bytes": 4.0 * (n * d + nq * d + nq) + 12.0 * nq * case["k"], "flops": 5.0 * nq * n * d}
    if do == "verify":
        nq, t = case["nq"], case["t"]
        return {"bytes": nq * (4.0 * t * d + 4 * t + 4 * d + 4 + 12 * case["k"]),
                "flops": 5.0 * nq * t * d}
    M = case["M"]
    if do == "build":
        rows = min(n, case["efc"] * M)
        return {"bytes": 4.0 * n * d + 8.0 * n * M, "flops": 3.0 * n * rows * d}
    nq, k, ef = case["nq"], case["k"] or 50, case["ef"] or 198
    rows = min(n, ef * M)
    return {"bytes": nq * (float(rows) * d * BYTES[case["dtype"]] + ef * 8.0 * M + 4.0 * ef * d
                           + 4 * d + 4 + 12 * k),
            "flops": nq * (3.0 * rows * d + 5.0 * ef * d)}


# ---------------------------------------------------------------- 64-bit answers
def _verify64(base, q, p, cand, k, mode):
    """Distances of the k nearest candidates; Algorithm 1 stops early, so that
    its answer is taken over the candidates it verified."""
    out = torch.empty((q.shape[0], k), dtype=torch.float64, device=DEV)
    t = cand.shape[1]
    step = max(1, (1 << 28) // (t * q.shape[1]))
    for s in range(0, q.shape[0], step):
        x = base[cand[s:s + step].long().reshape(-1)].view(-1, t, q.shape[1]).double()
        pp = p[s:s + step].double()
        S = (x - q[s:s + step, None].double()).abs_().pow_(pp[:, None, None]).sum(-1)
        if mode == "paper":
            taken = torch.full((S.shape[0],), t, device=DEV)
            open_ = torch.ones(S.shape[0], dtype=torch.bool, device=DEV)
            prev = torch.topk(S[:, :k], k, dim=1, largest=False).indices
            for i in range(k, t, k):
                end = min(i + k, t)
                new = torch.topk(S[:, :end], k, dim=1, largest=False).indices
                same = (new[:, :, None] == prev[:, None, :]).any(-1).sum(1)
                stop = open_ & (same.float() / k >= 0.92)
                taken[stop] = end
                open_ &= ~stop
                prev = new
            S = torch.where(torch.arange(t, device=DEV)[None] < taken[:, None], S, math.inf)
        S = torch.topk(S, k, dim=1, largest=False).values.sort(dim=1).values
        out[s:s + step] = S.pow(1.0 / pp[:, None])
    return out


def exact(case, seed):
    do, data, n, d = case["do"], case["data"], case["n"], case["d"]
    if do == "verify":
        q, cl, p = _queries(data, d, case["nq"], case["p"], seed)
        base = _base_dev(data, n, d)
        cand = _candidates(base, q, cl, n, case["t"], CLUSTERS[data])
        return None, _verify64(base, q, p, cand, case["k"], case["mode"])
    if do != "exact" or case["nq"] * float(n) * d > 2e11:
        return None
    q, _, p = _queries(data, d, case["nq"], case["p"], seed)
    base = _base_dev(data, n, d)
    k = min(case["k"], n)
    dist = torch.full((case["nq"], case["k"]), math.inf, dtype=torch.float64, device=DEV)
    pv = p.double().cpu().tolist()
    for i in range(case["nq"]):
        near = (base - q[i]).abs_().pow_(pv[i]).sum(1).topk(min(n, k + 64), largest=False).indices
        S = (base[near].double() - q[i].double()).abs_().pow_(pv[i]).sum(1)
        dist[i, :k] = S.topk(k, largest=False).values.sort().values.pow(1.0 / pv[i])
    return None, dist
