"""What the performance of this framework is measured on.

The cases are calls through the public entry points of ``paper_2411_06405_gb300``: whole
decompositions (normalise + peel) of a graph that has just arrived, h-support of a graph
that is kept, the CSR builder alone, batches of small graphs under both schedules, the
H-index iteration and the request loop.  Graph families and sizes are those of the
repository's workloads (Erdos-Renyi n = 2,000; R-MAT scale 16 and 18, edge factor 8; the
degree-corrected block model at n = 50,000 and 200,000; batches of ER and BA graphs; a
served mix of R-MAT and BA graphs) and the ranges between them.

Every output is an integer array that is fixed by the input alone.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2411_06405_gb300 as htd

RMAT = (0.57, 0.19, 0.19)  # quadrant probabilities a, b, c; d = 0.05
RAW = 1 + 1 / 16 + 1 / 64  # raw pairs per distinct edge: repeated pairs and loops included


# ---- inputs: raw undirected pairs, loops and duplicates included ------------------------

def _gen(seed: int, device) -> torch.Generator:
    g = torch.Generator(device=device)
    g.manual_seed(0x48545255 + seed)
    return g


def _er(n, k, gen, dev):
    return tuple(torch.randint(0, n, (k,), generator=gen, device=dev) for _ in range(2))


def _rmat(n, k, gen, dev):
    """Recursive-matrix pairs on 2**ceil(log2 n) ids, folded onto n ids."""
    scale = max(1, (n - 1).bit_length())
    a, b, c = RMAT
    s = torch.zeros(k, dtype=torch.int64, device=dev)
    d = torch.zeros(k, dtype=torch.int64, device=dev)
    for _ in range(scale):
        r = torch.rand(k, generator=gen, device=dev)
        s = 2 * s + (r >= a + b)
        d = 2 * d + (((r >= a) & (r < a + b)) | (r >= a + b + c))
    return (s * n) >> scale, (d * n) >> scale


def _dcsbm(n, k, gen, dev):
    """Degree-corrected block model: about n / 1,000 blocks of power-law sizes (exponent
    2.1), Pareto(2.5) degree propensities, 10% of the pairs between two random blocks."""
    blocks = max(4, n // 1000)
    f64 = {"dtype": torch.float64, "device": dev, "generator": gen}
    u = (torch.arange(blocks, device=dev, dtype=torch.float64) + 0.5) / blocks  # size quantiles
    cum = torch.cumsum(torch.clamp(100.0 * u ** (-1 / 1.1), max=0.1 * n), 0)
    bound = torch.floor(cum / cum[-1] * n).to(torch.int64)
    bound[-1] = n
    block = torch.searchsorted(bound, torch.arange(n, device=dev), right=True)
    cdf = torch.cumsum(torch.clamp(torch.rand(n, **f64) ** (-1 / 1.5), max=math.sqrt(n)), 0)
    top = cdf[torch.clamp(bound - 1, min=0)]
    low = torch.cat([torch.zeros(1, device=dev, dtype=torch.float64), top[:-1]])

    def vertex(blk):
        x = low[blk] + torch.rand(blk.numel(), **f64) * (top[blk] - low[blk])
        return torch.clamp(torch.searchsorted(cdf, x, right=True), max=n - 1)

    own = block[torch.randint(0, n, (k,), generator=gen, device=dev)]
    other = block[torch.randint(0, n, (k,), generator=gen, device=dev)]
    inter = torch.rand(k, generator=gen, device=dev) < 0.10
    return vertex(own), vertex(torch.where(inter, other, own))


def _ba(n, k, gen, dev):
    """Preferential attachment: every new vertex draws its targets from the endpoints of
    the earlier pairs.  A draw that hits an earlier target is resolved by pointer jumping."""
    src = (torch.arange(k, device=dev) * n) // k
    j = torch.arange(k, device=dev)
    # endpoint slots 0 .. 2j: slot 2i is the source of pair i, slot 2i + 1 its target
    pick = (torch.rand(k, generator=gen, device=dev, dtype=torch.float64) * (2 * j + 1)).to(torch.int64)
    while True:
        odd = (pick & 1) == 1
        if not bool(odd.any()):
            break
        pick = torch.where(odd, pick[pick >> 1], pick)
    return src, src[pick >> 1]


_FAMILY = {"er": _er, "rmat": _rmat, "dcsbm": _dcsbm, "ba": _ba}


def _pairs(family, n, edges, seed, dev="cuda"):
    """Raw pairs, int32, in random order: `edges` distinct undirected pairs, 1/16 of them
    once more and reversed, and edges // 64 loops."""
    gen = _gen(seed, dev)
    k = edges + edges // 8
    while True:
        s, d = _FAMILY[family](n, k, gen, dev)
        lo, hi = torch.minimum(s, d), torch.maximum(s, d)
        key = torch.unique((lo * n + hi)[lo != hi])
        if key.numel() >= edges:
            break
        k += max(edges // 4, 64)
    key = key[torch.randperm(key.numel(), generator=gen, device=dev)[:edges]]
    perm = torch.randperm(n, generator=gen, device=dev)
    u, v = perm[key // n], perm[key % n]
    again, loops = edges // 16, torch.randint(0, n, (edges // 64,), generator=gen, device=dev)
    s, d = torch.cat([u, v[:again], loops]), torch.cat([v, u[:again], loops])
    order = torch.randperm(s.numel(), generator=gen, device=dev)
    return s[order].to(torch.int32).contiguous(), d[order].to(torch.int32).contiguous()


def _mixed_graphs(count, n_lo, n_hi, seed):
    """A batch: n uniform in [n_lo, n_hi], ER of mean degree 8 or BA, h in {2, 3}.  The
    seed draws the edges; sizes and kinds belong to the case."""
    rng = np.random.default_rng(7 * count + n_hi)
    out = []
    for i in range(count):
        n, h = int(rng.integers(n_lo, n_hi + 1)), int(rng.integers(2, 4))
        fam, deg = ("er", 4) if rng.random() < 0.5 else ("ba", int(rng.integers(2, 9)))
        s, d = _pairs(fam, n, deg * n, 4096 * seed + i, "cpu")
        out.append((n, s.numpy(), d.numpy(), h))
    return out


def _requests(count, n_lo, n_hi, seed):
    """A burst of requests: R-MAT (edge factor 7) or BA, n log-uniform, h in {2, 3}."""
    rng = np.random.default_rng(7 * count + n_hi)
    out = []
    for i in range(count):
        n = int(round(math.exp(rng.uniform(math.log(n_lo), math.log(n_hi)))))
        fam, deg = ("rmat", 7) if rng.random() < 0.5 else ("ba", int(rng.integers(2, 9)))
        s, d = _pairs(fam, n, deg * n, 4096 * seed + i, "cpu")
        out.append((n, s.numpy(), d.numpy(), int(rng.integers(2, 4))))
    return out


# ---- the cases --------------------------------------------------------------------------

def listed():
    return [
        # a small graph decomposed as it arrives: launches and latency are all of it
        {"name": "peel_er_n2000_h2", "op": "peel", "family": "er", "n": 2000, "edges": 8000, "h": 2},
        # a power-law graph with hubs: long h-hop rows beside short ones
        {"name": "peel_rmat_s16_h2", "op": "peel", "family": "rmat", "n": 65536, "edges": 477437, "h": 2},
        # a large social-like graph; with the removal rounds that a certificate needs
        {"name": "peel_dcsbm_n200k_h2", "op": "peel_stamps", "family": "dcsbm", "n": 200000,
         "edges": 1200000, "h": 2},
        # radius 3: the rounds that keep two ball sets
        {"name": "peel_dcsbm_n40k_h3", "op": "peel", "family": "dcsbm", "n": 40000, "edges": 240000, "h": 3},
        # the classic truss (h = 1), end to end through host buffers
        {"name": "host_rmat_s16_h1", "op": "host", "family": "rmat", "n": 65536, "edges": 477437, "h": 1},
        # h-support alone on a kept graph: hub rows at radius 2, many members at radius 3
        {"name": "support_rmat_s18_h2", "op": "support", "family": "rmat", "n": 262144, "edges": 1969330, "h": 2},
        {"name": "support_dcsbm_n200k_h3", "op": "support", "family": "dcsbm", "n": 200000,
         "edges": 1200000, "h": 3},
        # normalisation of raw pairs alone
        {"name": "csr_rmat_s18", "op": "csr", "family": "rmat", "n": 262144, "edges": 1969330, "h": 0},
        # many graphs in one call: concurrent unions, and one block per small graph
        {"name": "batch_64_n50_5000", "op": "batch", "count": 64, "n_lo": 50, "n_hi": 5000},
        {"name": "blocks_256_n50_600", "op": "blocks", "count": 256, "n_lo": 50, "n_hi": 600},
        # the H-index iteration with pruning, the second engine
        {"name": "hindex_dcsbm_n50k_h2", "op": "hindex", "family": "dcsbm", "n": 50000, "edges": 300000, "h": 2},
        # a burst of requests to a running server
        {"name": "served_12_n1k_8k", "op": "served", "count": 12, "n_lo": 1000, "n_hi": 8000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["peel"] * 5 + ["peel_stamps", "host", "host", "support", "support", "csr", "batch",
                                    "blocks", "hindex", "served"])
    if op in ("batch", "blocks"):
        hi = _log_int(rng, 300, 5000) if op == "batch" else _log_int(rng, 100, 600)
        return {"op": op, "count": _log_int(rng, 4, 64 if op == "batch" else 256), "n_lo": 50, "n_hi": hi}
    if op == "served":
        return {"op": op, "count": rng.randint(2, 12), "n_lo": 1000, "n_hi": _log_int(rng, 2000, 8000)}
    family = rng.choice(["er", "rmat", "dcsbm", "ba"])
    if op == "csr":
        n, h = _log_int(rng, 1000, 262144), 0
    elif op == "support":
        h = rng.choice([1, 2, 3])
        n = _log_int(rng, 1000, 200000 if h < 3 else 50000)
    elif op == "hindex":
        h, n = 2, _log_int(rng, 1000, 20000)
    else:
        h = rng.choice([1, 2, 2, 3])
        n = _log_int(rng, 500, {1: 65536, 2: 40000, 3: 8000}[h])
    degree = 7 if family == "rmat" else 4 if family == "er" else rng.randint(2, 6)
    return {"op": op, "family": family, "n": n, "edges": degree * n + rng.randint(0, 7), "h": h}


def prepare(case, seed):
    op = case["op"]
    if op in ("batch", "blocks"):
        graphs = _mixed_graphs(case["count"], case["n_lo"], case["n_hi"], seed)
        return {"op": op, "batch": htd.BatchInput(graphs),
                "flags": htd.HTD_OPT_BATCH_BLOCKS if op == "blocks" else 0}
    if op == "served":
        return {"op": op, "requests": _requests(case["count"], case["n_lo"], case["n_hi"], seed),
                "server": htd.Server(workers=4)}
    s, d = _pairs(case["family"], case["n"], case["edges"], seed)
    st = {"op": op, "n": case["n"], "h": case["h"], "src": s, "dst": d}
    if op == "host":
        k = s.numel()
        st["src"], st["dst"] = s.cpu().pin_memory(), d.cpu().pin_memory()
        st["out"] = [torch.empty(k, dtype=torch.int32).pin_memory() for _ in range(3)]
    elif op in ("support", "hindex"):
        st["graph"] = htd.htd_build_csr(case["n"], s, d)
    return st


def run(state):
    op = state["op"]
    if op in ("peel", "peel_stamps"):
        g = htd.htd_build_csr(state["n"], state["src"], state["dst"])
        truss, stamp, _ = htd.htd_truss_decompose(g, state["h"], stamps=op == "peel_stamps")
        eu, ev = htd.htd_edges(g)
        return {"eu": eu, "ev": ev, "truss": truss, **({} if stamp is None else {"stamp": stamp})}
    if op == "host":
        eu, ev, truss, _ = htd.htd_truss_decompose_host(state["n"], state["src"], state["dst"], state["h"],
                                                        *state["out"])
        return {"eu": eu, "ev": ev, "truss": truss}
    if op == "support":
        return htd.htd_h_support(state["graph"], state["h"])
    if op == "csr":
        g = htd.htd_build_csr(state["n"], state["src"], state["dst"])
        row_ptr, col, eid = htd.htd_csr(g)
        eu, ev = htd.htd_edges(g)
        return {"row_ptr": row_ptr, "col": col, "eid": eid, "eu": eu, "ev": ev}
    if op in ("batch", "blocks"):
        # the graphs' results are consecutive views of the batch's own output buffer
        res, _ = htd.htd_truss_decompose_batched(state["batch"], flags=state["flags"])
        return {"truss": torch.cat(res), "m": torch.tensor([r.numel() for r in res])}
    if op == "hindex":
        truss, hval, _ = htd.htd_hindex_decompose(state["graph"], state["h"], prune=True)
        return {"truss": truss, "hval": hval}
    server = state["server"]
    ids = [server.submit(n, s, d, h) for n, s, d, h in state["requests"]]
    got = [server.wait(i, r[1].size) for i, r in zip(ids, state["requests"])]
    return {k: np.concatenate([g[j] for g in got]) for j, k in enumerate(("eu", "ev", "truss"))}


def work(case):
    """Bytes only (nothing here is a floating-point operation): the raw pairs read once and
    the outputs written once."""
    op = case["op"]
    if op in ("batch", "blocks", "served"):
        n = ((case["n_lo"] + case["n_hi"]) / 2 if op != "served"
             else (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"]))
        k = case["count"] * n * (4.5 if op != "served" else 6)  # mean edges per vertex
        return {"bytes": k * (RAW * 8 + (4 if op != "served" else 12))}
    k = case["edges"]
    per = {"peel": 12, "peel_stamps": 16, "host": 12, "support": 4, "hindex": 8, "csr": 24}[op]
    return {"bytes": k * (RAW * 8 + per) + (4 * (case["n"] + 1) if op == "csr" else 0)}


# ---- the same values by dense linear algebra and sorting, without the framework ---------

def _dense_balls(adj, h):
    ball = reach = adj + torch.eye(adj.shape[0], dtype=adj.dtype, device=adj.device)
    for _ in range(h - 1):
        ball = ((ball @ reach) > 0).to(adj.dtype)
    return ball


def _dense_support(adj, u, v, h):
    ball = _dense_balls(adj, h)
    return (ball @ ball)[u, v].round().to(torch.int64) - 2


def exact(case, seed):
    op = case["op"]
    if op not in ("peel", "support", "csr") or (op != "csr" and case["n"] > 2500):
        return None
    n = case["n"]
    s, d = (x.to(torch.int64) for x in _pairs(case["family"], n, case["edges"], seed))
    lo, hi = torch.minimum(s, d), torch.maximum(s, d)
    key = torch.unique((lo * n + hi)[lo != hi])
    u, v = key // n, key % n
    m = u.numel()
    if op == "csr":
        slot = torch.cat([u * n + v, v * n + u])
        slot, order = torch.sort(slot)
        eid = torch.cat([torch.arange(m, device=u.device)] * 2)[order]
        row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=u.device)
        row_ptr[1:] = torch.cumsum(torch.bincount(slot // n, minlength=n), 0)
        got = {"row_ptr": row_ptr, "col": slot % n, "eid": eid, "eu": u, "ev": v}
        return {k: x.to(torch.int32) for k, x in got.items()}
    adj = torch.zeros(n, n, dtype=torch.float64, device=u.device)
    adj[u, v] = adj[v, u] = 1.0
    if op == "support":
        return _dense_support(adj, u, v, case["h"]).to(torch.int32)
    truss = torch.zeros(m, dtype=torch.int32, device=u.device)
    alive, k = torch.ones(m, dtype=torch.bool, device=u.device), 2
    if n * case["h"] > 6000:
        return None
    while bool(alive.any()):
        sup = _dense_support(adj, u, v, case["h"])
        k = max(k, int(sup[alive].min()) + 2)
        gone = alive & (sup <= k - 2)
        truss[gone] = k
        adj[u[gone], v[gone]] = adj[v[gone], u[gone]] = 0.0
        alive &= ~gone
    return {"eu": u.to(torch.int32), "ev": v.to(torch.int32), "truss": truss}
