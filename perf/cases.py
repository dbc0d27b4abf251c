"""The measured workloads of the framework: what its users have it do, over the
sizes they do it at.

A case is a dict of plain values with a "kind":
  pagerank  20 iterations on a graph that is already clustered and segmented
            ("path": "plan" the GPU plan after clustering, "uniform" the
            paper's equal split into "k" segments in the graph's own
            numbering, "plain" the unsegmented pull, "one" one personalised
            vector on the plan)
  solve     a graph nobody has seen: clustering, segmenting and 20 iterations
  lp        label propagation on an undirected graph until nothing changes
  ppr       64 personalised vectors in one gather ("hubs": the size of the
            dense hub block on the tensor cores, 0 for none)
  cf        sweeps of collaborative filtering on a rating matrix ("precision"
            "f32" or "hilo"; plain BF16 storage is left out: steps of 1e-3
            round away in it, so nobody trains with it)
  batch     PageRank of many small graphs in one launch
  bc        betweenness centrality from a few sources

Inputs are synthetic and made on the GPU from the seed: RMAT graphs
(a, b, c, d = 0.57, 0.19, 0.19, 0.05; self-loops and duplicate edges dropped,
vertices shuffled) of any number of vertices, and rating matrices with
lognormal user activity and Zipf item popularity.
"""
import math
import random

import numpy as np
import torch

from paper_1608_01362_gb300 import cagra as C
from paper_1608_01362_gb300 import pipeline as P

DEV = "cuda"
ITERS = 20
DAMPING = 0.85
LAMBDA, STEP, SWEEPS = 0.05, 1e-3, 10
PRECISION = {"f32": C.CF_FP32, "hilo": C.CF_BF16X2}
MIN_DEGREE = 32.0   # head threshold of the GPU plan (the autotuner's usual pick)
LP_PASSES = 7       # passes an undirected RMAT graph takes, for work()


def listed():
    return [
        # a graph of a test or of one community: 20 iterations are 80 launches
        {"name": "pagerank_small", "kind": "pagerank", "path": "plan", "V": 20011, "E": 300_000},
        # an everyday graph, edges and vertex arrays within the L2
        {"name": "pagerank_mid", "kind": "pagerank", "path": "plan", "V": 1 << 20,
         "E": 15_700_000},
        # the benchmark's graph: the size of the paper's RMAT and Twitter inputs
        {"name": "pagerank_large", "kind": "pagerank", "path": "plan", "V": 1 << 25,
         "E": 528_688_805},
        # a graph that is solved once: clustering and segmenting count
        {"name": "solve_mid", "kind": "solve", "V": 1 << 22, "E": 65_242_799},
        # connected components of an undirected graph
        {"name": "lp_mid", "kind": "lp", "V": 3_000_017, "E": 96_000_000},
        # recommendations for 64 users at once
        {"name": "ppr_mid", "kind": "ppr", "V": 1 << 20, "E": 15_700_000, "hubs": 0},
        # the Netflix-shaped matrix of the paper's Table III, in hi + lo storage
        {"name": "cf_large", "kind": "cf", "U": 480_189, "I": 17_770, "R": 99_000_000, "K": 32,
         "precision": "hilo"},
        # a shop's or a film club's matrix, wider factors in FP32
        {"name": "cf_small", "kind": "cf", "U": 30_011, "I": 4_001, "R": 2_000_003, "K": 64,
         "precision": "f32"},
        # a collection of small graphs (ego networks, molecules, documents)
        {"name": "batch_large", "kind": "batch", "G": 1024, "lo": 8, "hi": 15, "deg": 16},
        # a handful of them: fewer graphs than the GPU has SMs
        {"name": "batch_small", "kind": "batch", "G": 40, "lo": 8, "hi": 12, "deg": 16},
        # the paper's 12 sources
        {"name": "bc_large", "kind": "bc", "V": 1 << 22, "E": 65_242_799, "sources": 12},
        # a few sources on a small graph: many short levels
        {"name": "bc_small", "kind": "bc", "V": 65_537, "E": 900_000, "sources": 4},
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["pagerank", "pagerank", "pagerank", "solve", "lp", "ppr", "cf", "cf",
                       "batch", "bc"])
    if kind == "pagerank":
        path = rng.choice(["plan", "plan", "plan", "uniform", "one", "plain"])
        V = _log(rng, 4_000, 30_000_000)
        c = {"kind": kind, "path": path, "V": V, "E": _edges(rng, V, 400_000_000)}
        if path == "uniform":
            c["k"] = rng.choice([1, 3, 4, 8, 16])
        return c
    if kind == "solve":
        V = _log(rng, 10_000, 16_000_000)
        return {"kind": kind, "V": V, "E": _edges(rng, V, 200_000_000)}
    if kind == "lp":
        V = _log(rng, 10_000, 10_000_000)
        return {"kind": kind, "V": V, "E": _edges(rng, V, 200_000_000)}
    if kind == "ppr":
        V = _log(rng, 10_000, 4_000_000)
        return {"kind": kind, "V": V, "E": _edges(rng, V, 60_000_000),
                "hubs": 4096 if V > 100_000 and rng.random() < 0.25 else 0}
    if kind == "cf":
        U = _log(rng, 2_000, 400_000)
        I = _log(rng, 500, 30_000)
        R = min(int(U * rng.uniform(20, 200)), U * I // 20, 80_000_000)
        return {"kind": kind, "U": U, "I": I, "R": R, "K": rng.choice([16, 32, 32, 64]),
                "precision": rng.choice(["f32", "hilo"])}
    if kind == "batch":
        lo = rng.randint(6, 10)
        return {"kind": kind, "G": _log(rng, 8, 1000), "lo": lo, "hi": rng.randint(lo, 14),
                "deg": rng.randint(4, 16)}
    V = _log(rng, 10_000, 8_000_000)
    return {"kind": kind, "V": V, "E": _edges(rng, V, 100_000_000),
            "sources": rng.randint(1, 12)}


def _edges(rng, V, most):
    return min(int(V * rng.uniform(6, 24)), most)


# ------------------------------------------------------------------ inputs


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)


def _rmat_pairs(n, scale, g):
    """n RMAT edges (source, destination) over 2^scale IDs."""
    src = torch.zeros(n, dtype=torch.int32, device=DEV)
    dst = torch.zeros(n, dtype=torch.int32, device=DEV)
    for _ in range(scale):
        r = torch.rand(n, device=DEV, generator=g)
        s = r >= 0.76
        src.mul_(2).add_(s)
        dst.mul_(2).add_((r >= 0.95) | ((r >= 0.57) & ~s))
    return src, dst


def _rmat_keys(V, E, g, symmetric=False):
    """E distinct edges as sorted keys destination * V + source; an odd number
    of undirected edges leaves one short."""
    scale = max(1, (V - 1).bit_length())
    perm = torch.randperm(V, device=DEV, generator=g, dtype=torch.int32)
    want = E // 2 if symmetric else E
    have = None
    while have is None or have.numel() < want:
        missing = want - (0 if have is None else have.numel())
        src, dst = _rmat_pairs(int(1.15 * missing) + 64, scale, g)
        if V != 1 << scale:
            src = ((src.long() * V) >> scale).int()
            dst = ((dst.long() * V) >> scale).int()
        src, dst = perm[src], perm[dst]
        keep = src != dst
        src, dst = src[keep], dst[keep]
        if symmetric:  # one direction stands for both
            src, dst = torch.minimum(src, dst), torch.maximum(src, dst)
        key = dst.long() * V + src
        del src, dst, keep
        have = torch.unique(key if have is None else torch.cat([have, key]))
        del key
    n = have.numel()
    if n > want:  # drop the surplus evenly over the sorted keys
        mask = torch.ones(n, dtype=torch.bool, device=DEV)
        mask[(torch.arange(n - want, device=DEV) * n) // (n - want)] = False
        have = have[mask]
    if symmetric:
        have = torch.cat([have, (have % V) * V + have // V]).sort().values
    return have


def _graph(V, E, seed, symmetric=False):
    """In-edge CSR (offsets int64 [V+1], sources int32) and its generator."""
    g = _gen(seed)
    key = _rmat_keys(V, E, g, symmetric)
    deg = torch.bincount(key // V, minlength=V)
    off = torch.zeros(V + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(deg, 0, out=off[1:])
    return off, (key % V).int(), g


def _vertices(src, V, n, g):
    """n distinct vertices that have out-edges, as a list."""
    have = torch.nonzero(torch.bincount(src, minlength=V)).flatten()
    at = torch.randperm(have.numel(), device=DEV, generator=g)[:n]
    return have[at].tolist()


def _batch(case, seed):
    """Many small RMAT graphs end to end: (vbase, offsets, local sources)."""
    g = _gen(seed)
    rng = random.Random(case["G"])  # the sizes are the case's, the edges the seed's
    scale = np.array([rng.randint(case["lo"], case["hi"]) for _ in range(case["G"])])
    vbase = np.concatenate([[0], np.cumsum(1 << scale)]).astype(np.int64)
    V = int(vbase[-1])
    base = torch.from_numpy(vbase[:-1]).to(DEV)
    bits = torch.from_numpy(scale).to(DEV)
    gid = torch.repeat_interleave(torch.arange(case["G"], device=DEV), case["deg"] << bits)
    n = gid.numel()
    lev = bits.int()[gid]
    src = torch.zeros(n, dtype=torch.int32, device=DEV)
    dst = torch.zeros(n, dtype=torch.int32, device=DEV)
    for b in range(int(scale.max())):
        r = torch.rand(n, device=DEV, generator=g)
        on = lev > b
        s = r >= 0.76
        src += (on & s).int() << b
        dst += (on & ((r >= 0.95) | ((r >= 0.57) & ~s))).int() << b
    # shuffle the IDs inside each graph
    vg = torch.repeat_interleave(torch.arange(case["G"], device=DEV), 1 << bits)
    order = torch.argsort(vg + torch.rand(V, device=DEV, generator=g, dtype=torch.float64))
    place = torch.empty(V, dtype=torch.int64, device=DEV)
    place[order] = torch.arange(V, device=DEV)
    src, dst = place[base[gid] + src], place[base[gid] + dst]
    keep = src != dst
    key = torch.unique(dst[keep] * V + src[keep])
    dst, src = key // V, key % V
    off = torch.zeros(V + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(dst, minlength=V), 0, out=off[1:])
    return vbase, off, (src - base[vg[src]]).int(), src


def _ratings(case, seed):
    """User-major rating CSR (offsets, items int32, ratings uint8) and FP32
    factors: lognormal user activity, Zipf item popularity, no pair twice."""
    g = _gen(seed)
    U, I, R, K = case["U"], case["I"], case["R"], case["K"]
    act = torch.exp(1.2 * torch.randn(U, device=DEV, generator=g, dtype=torch.float64))
    act = torch.cumsum(act.clamp_(max=act.mean() * 0.2 * I * U / R), 0)
    pop = torch.cumsum(1.0 / torch.arange(1, I + 1, device=DEV, dtype=torch.float64), 0)
    item = torch.randperm(I, device=DEV, generator=g)
    have = None
    while have is None or have.numel() < R:
        missing = R - (0 if have is None else have.numel())
        n = 2 * missing + 64  # the hottest items repeat
        ru = torch.rand(n, device=DEV, generator=g, dtype=torch.float64) * act[-1]
        ri = torch.rand(n, device=DEV, generator=g, dtype=torch.float64) * pop[-1]
        u = torch.searchsorted(act, ru).clamp_(max=U - 1)
        i = item[torch.searchsorted(pop, ri).clamp_(max=I - 1)]
        key = u * I + i
        del ru, ri, u, i
        have = torch.unique(key if have is None else torch.cat([have, key]))
        del key
    n = have.numel()
    if n > R:
        mask = torch.ones(n, dtype=torch.bool, device=DEV)
        mask[(torch.arange(n - R, device=DEV) * n) // (n - R)] = False
        have = have[mask]
    off = torch.zeros(U + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(have // I, minlength=U), 0, out=off[1:])
    rate = torch.randint(1, 6, (R,), device=DEV, generator=g, dtype=torch.uint8)
    hi = math.sqrt(12.0 / K)
    Pf = torch.rand(U, K, device=DEV, generator=g) * hi
    Qf = torch.rand(I, K, device=DEV, generator=g) * hi
    return off, (have % I).int(), rate, Pf, Qf


# ------------------------------------------------------------------ the passes


def _planned(graph):
    return P.SegmentedPageRank(graph, bounds=P.plan_bounds(graph, min_avg_degree=MIN_DEGREE))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pagerank":
        off, src, g = _graph(case["V"], case["E"], seed)
        if case["path"] == "plain":
            return {"kind": kind, "pr": P.PlainPageRank(P.Graph(off, src, cluster_mode=None))}
        if case["path"] == "uniform":
            graph = P.Graph(off, src, cluster_mode=None)
            return {"kind": kind, "pr": P.SegmentedPageRank(graph, case["k"])}
        state = {"kind": kind, "pr": _planned(P.Graph(off, src, cluster_mode=0))}
        if case["path"] == "one":
            state |= {"kind": "one", "seed": _vertices(src, case["V"], 1, g)[0]}
        return state
    if kind == "solve":
        off, src, _ = _graph(case["V"], case["E"], seed)
        return {"kind": kind, "off": off, "src": src}
    if kind == "lp":
        off, src, _ = _graph(case["V"], case["E"], seed, symmetric=True)
        graph = P.Graph(off, src, cluster_mode=0)
        bounds = P.plan_bounds(graph, min_avg_degree=24.0)
        return {"kind": kind, "lp": P.LabelPropagation(graph, bounds=bounds)}
    if kind == "ppr":
        off, src, g = _graph(case["V"], case["E"], seed)
        ppr = P.BatchedPPR(P.Graph(off, src, cluster_mode=0), 1, dense_hubs=case["hubs"])
        return {"kind": kind, "ppr": ppr, "seeds": _vertices(src, case["V"], C.PPR_COLUMNS, g)}
    if kind == "cf":
        off, item, rate, Pf, Qf = _ratings(case, seed)
        U, I = case["U"], case["I"]
        ioff = torch.empty(I + 1, dtype=torch.int64, device=DEV)
        iuser, irate = torch.empty_like(item), torch.empty_like(rate)
        C.cf_transpose(U, I, off, item, rate, ioff, iuser, irate)
        cf = C.cf_create(U, I, case["K"], PRECISION[case["precision"]], off, item, rate, ioff,
                         iuser, irate)
        return {"kind": kind, "cf": cf, "P": Pf, "Q": Qf, "P1": torch.empty_like(Pf),
                "Q1": torch.empty_like(Qf),
                "sse": torch.zeros(SWEEPS, dtype=torch.float64, device=DEV)}
    if kind == "batch":
        vbase, off, src, _ = _batch(case, seed)
        return {"kind": kind, "b": C.pr_batch_create(vbase, off, src),
                "rank": torch.empty(int(vbase[-1]), dtype=torch.float32, device=DEV)}
    off, src, g = _graph(case["V"], case["E"], seed)
    sources = _vertices(src, case["V"], case["sources"], g)
    return {"kind": kind, "bc": P.Betweenness(P.Graph(off, src, cluster_mode=0)),
            "sources": sources}


def run(state):
    # residuals and squared errors are FP64 sums of FP32 terms: handed on in FP32
    kind = state["kind"]
    if kind == "pagerank":
        rank, resid = state["pr"].run(ITERS, DAMPING)
        return {"rank": rank, "resid": resid.float()}
    if kind == "one":
        rank, resid = state["pr"].run_ppr(state["seed"], ITERS, DAMPING)
        return {"rank": rank, "resid": resid.float()}
    if kind == "solve":
        rank, resid = _planned(P.Graph(state["off"], state["src"], cluster_mode=0)).run(ITERS,
                                                                                        DAMPING)
        return {"rank": rank, "resid": resid.float()}
    if kind == "lp":
        labels, passes, changes = state["lp"].run()
        return {"labels": labels, "passes": passes, "changes": changes}
    if kind == "ppr":
        # 20 iterations converge: the residual of the last one is rounding alone
        rank, _ = state["ppr"].run(state["seeds"], ITERS, DAMPING)
        return {"rank": rank}
    if kind == "cf":
        cf = state["cf"]
        C.cf_set_factors(cf, state["P"], state["Q"])
        C.cf_sweep(cf, SWEEPS, LAMBDA, STEP, state["sse"])
        C.cf_get_factors(cf, state["P1"], state["Q1"])
        return {"P": state["P1"], "Q": state["Q1"], "sse": state["sse"].float()}
    if kind == "batch":
        C.pr_batch_run(state["b"], ITERS, DAMPING, state["rank"])
        return {"rank": state["rank"]}
    return {"bc": state["bc"].run(state["sources"])}


def work(case):
    """Bytes and operations of one pass: per iteration, pass, sweep or search
    the edges (4 bytes each) and the vertex arrays once."""
    kind = case["kind"]
    if kind in ("pagerank", "solve"):
        V, E = case["V"], case["E"]
        b = ITERS * (4 * E + 28 * V)
        if kind == "solve":  # the CSR in, renumbered, and segmented
            b += 3 * (4 * E + 8 * V) + 16 * V
        return {"bytes": b, "flops": ITERS * (E + 5 * V)}
    if kind == "lp":
        return {"bytes": LP_PASSES * (4 * case["E"] + 20 * case["V"]),
                "flops": LP_PASSES * case["E"]}
    if kind == "ppr":
        V, E, n = case["V"], case["E"], C.PPR_COLUMNS
        return {"bytes": ITERS * (4 * E + 12 * V + 2 * 4 * n * V) + 4 * n * V,
                "flops": ITERS * n * (E + 2 * V)}
    if kind == "cf":
        U, I, R, K = case["U"], case["I"], case["R"], case["K"]
        return {"bytes": SWEEPS * (2 * 5 * R + 8 * (U + I) + 2 * 4 * K * (U + I)),
                "flops": SWEEPS * R * (6 * K + 3)}
    if kind == "batch":
        V = case["G"] * sum(1 << s for s in range(case["lo"], case["hi"] + 1)) \
            // (case["hi"] - case["lo"] + 1)
        E = V * case["deg"]
        return {"bytes": ITERS * (4 * E + 12 * V), "flops": ITERS * (E + 5 * V)}
    V, E = case["V"], case["E"]
    return {"bytes": case["sources"] * (2 * 4 * E + 56 * V), "flops": case["sources"] * 2 * E}


# ------------------------------------------------------------------ 64-bit values


def _csr(off, src, values, cols):
    return torch.sparse_csr_tensor(off.int(), src, values, size=(off.numel() - 1, cols),
                                   dtype=torch.float64, device=DEV)


def _ones(src):
    return torch.ones(src.numel(), dtype=torch.float64, device=DEV)


def _iterate(A, outdeg, r, tele):
    """ITERS iterations of the normalised update from r; tele: where the
    teleport and the dangling mass go (columns that sum to 1)."""
    inv = torch.where(outdeg > 0, 1.0 / outdeg.clamp(min=1).double(), 0.0)
    dang = (outdeg == 0).double()
    if r.dim() == 2:
        inv, dang = inv[:, None], dang[:, None]
    resid = []
    for _ in range(ITERS):
        D = (dang * r).sum(0)
        new = DAMPING * (A @ (r * inv)) + tele * ((1 - DAMPING) + DAMPING * D)
        resid.append((new - r).abs().sum(0))
        r = new
    return r, torch.stack(resid)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pagerank", "solve"):
        V = case["V"]
        off, src, g = _graph(V, case["E"], seed)
        outdeg = torch.bincount(src, minlength=V)
        if case.get("path") == "one":
            tele = torch.zeros(V, dtype=torch.float64, device=DEV)
            tele[_vertices(src, V, 1, g)[0]] = 1.0
            r = tele.clone()
        else:
            tele = torch.full((V,), 1.0 / V, dtype=torch.float64, device=DEV)
            r = tele.clone()
        r, resid = _iterate(_csr(off, src, _ones(src), V), outdeg, r, tele)
        return {"rank": r, "resid": resid}
    if kind == "lp":
        V = case["V"]
        off, src, _ = _graph(V, case["E"], seed, symmetric=True)
        dst = torch.repeat_interleave(torch.arange(V, device=DEV), off[1:] - off[:-1])
        lab, changes = torch.arange(V, device=DEV, dtype=torch.int32), []
        while not changes or changes[-1]:
            new = lab.scatter_reduce(0, dst, lab[src], "amin")
            changes.append(int((new != lab).sum()))
            lab = new
        return {"labels": lab, "passes": len(changes), "changes": np.array(changes)}
    if kind == "ppr":
        V, n = case["V"], C.PPR_COLUMNS
        off, src, g = _graph(V, case["E"], seed)
        tele = torch.zeros(V, n, dtype=torch.float64, device=DEV)
        tele[_vertices(src, V, n, g), list(range(n))] = 1.0
        outdeg = torch.bincount(src, minlength=V)
        r, _ = _iterate(_csr(off, src, _ones(src), V), outdeg, tele.clone(), tele)
        return {"rank": r}
    if kind == "cf":
        return _exact_cf(case, seed)
    if kind == "batch":
        vbase, off, _, src = _batch(case, seed)
        V = int(vbase[-1])
        n = torch.from_numpy(np.diff(vbase)).to(DEV)
        gid = torch.repeat_interleave(torch.arange(case["G"], device=DEV), n)
        outdeg = torch.bincount(src, minlength=V)
        inv = torch.where(outdeg > 0, 1.0 / outdeg.clamp(min=1).double(), 0.0)
        A = _csr(off, src.int(), _ones(src), V)
        share = (1.0 / n.double())[gid]
        r = share.clone()
        for _ in range(ITERS):
            D = torch.zeros(case["G"], dtype=torch.float64, device=DEV)
            D.index_add_(0, gid, torch.where(outdeg == 0, r, 0.0))
            r = DAMPING * (A @ (r * inv)) + share * ((1 - DAMPING) + DAMPING * D[gid])
        return {"rank": r}
    return {"bc": _exact_bc(case, seed)}


def _exact_cf(case, seed):
    off, item, rate, Pf, Qf = _ratings(case, seed)
    U, I = case["U"], case["I"]
    p, q = Pf.double(), Qf.double()
    user = torch.repeat_interleave(torch.arange(U, device=DEV, dtype=torch.int32),
                                   off[1:] - off[:-1])
    order = torch.argsort(item, stable=True)
    ioff = torch.zeros(I + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(item, minlength=I), 0, out=ioff[1:])
    iuser = user[order]
    du = (off[1:] - off[:-1]).clamp(min=1).double()[:, None]
    di = (ioff[1:] - ioff[:-1]).clamp(min=1).double()[:, None]
    sse = []
    for _ in range(SWEEPS):
        e = torch.empty(item.numel(), dtype=torch.float64, device=DEV)
        for a in range(0, item.numel(), 4_000_000):
            s = slice(a, a + 4_000_000)
            e[s] = rate[s] - (p[user[s]] * q[item[s]]).sum(1)
        sse.append((e * e).sum())
        gp = _csr(off, item, e, I) @ q
        gq = _csr(ioff, iuser, e[order], U) @ p
        p, q = p + STEP * (gp / du - LAMBDA * p), q + STEP * (gq / di - LAMBDA * q)
    return {"P": p, "Q": q, "sse": torch.stack(sse)}


def _exact_bc(case, seed):
    V = case["V"]
    off, src, g = _graph(V, case["E"], seed)
    sources = _vertices(src, V, case["sources"], g)
    A = _csr(off, src, _ones(src), V)  # row = destination
    dst = torch.repeat_interleave(torch.arange(V, device=DEV, dtype=torch.int32),
                                  off[1:] - off[:-1])
    out_off = torch.zeros(V + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(src, minlength=V), 0, out=out_off[1:])
    out = _csr(out_off, dst[torch.argsort(src, stable=True)], _ones(src), V)
    bc = torch.zeros(V, dtype=torch.float64, device=DEV)
    for s in sources:
        level = torch.full((V,), -1, dtype=torch.int32, device=DEV)
        sigma = torch.zeros(V, dtype=torch.float64, device=DEV)
        level[s], sigma[s], depth = 0, 1.0, 0
        while True:
            y = A @ torch.where(level == depth, sigma, 0.0)
            new = (y > 0) & (level < 0)
            if not bool(new.any()):
                break
            depth += 1
            level[new] = depth
            sigma = torch.where(new, y, sigma)
        delta = torch.zeros(V, dtype=torch.float64, device=DEV)
        for d in range(depth - 1, -1, -1):
            y = out @ torch.where(level == d + 1, (1 + delta) / sigma.clamp(min=1), 0.0)
            delta = torch.where(level == d, sigma * y, delta)
        delta[s] = 0.0
        bc += delta
    return bc
