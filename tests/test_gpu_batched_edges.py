"""Batched PageRank at the edges of its layout: rows of more than one and two
full tasks (4096 edges), graphs whose row sums fit on chip next to graphs whose
do not, the largest graph a block can hold, sources outside their graph, with
and without residuals.  Every rank within the oracle's rounding bound."""
import numpy as np
import pytest

import graphgen
import oracle as O
from parity import check_pagerank

pytestmark = pytest.mark.gpu


def _star(n, k):
    """k vertices that every other one points at, and a cycle."""
    hub = np.arange(k)
    s = np.concatenate([np.tile(np.arange(n), k), np.arange(n)])
    d = np.concatenate([np.repeat(hub, n), (np.arange(n) + 1) % n])
    return graphgen.from_edges(n, s, d)


SETS = {
    "hubs": lambda: [_star(9001, 3), _star(4097, 1), _star(4098, 2), graphgen.rmat(7, 8, seed=2)],
    "mixed": lambda: [_star(40_000, 1)] + [graphgen.rmat(s, 6, seed=s) for s in (14, 15, 13, 5)],
    "largest": lambda: [_star(57_599, 1), _star(57_600, 0), graphgen.from_edges(3, [0], [1])],
}


@pytest.mark.parametrize("threads", [1024, 512, 256])
@pytest.mark.parametrize("name", list(SETS))
def test_ranks_and_residuals(name, threads):
    import torch
    from paper_1608_01362_gb300 import pipeline as P
    gs = SETS[name]()
    bp = P.BatchedPageRank(gs, threads=threads)
    resid = torch.zeros(len(gs) * 8, dtype=torch.float64, device="cuda")
    with_resid = bp.run(8, resid=resid).clone()
    plain = bp.run(8).clone()
    assert torch.equal(plain, with_resid) and torch.equal(bp.run(8), plain)
    rank = plain.cpu().numpy()
    res = resid.cpu().numpy().reshape(len(gs), 8)
    for i, g in enumerate(gs):
        wres = np.zeros(8)
        want, bound = O.pagerank_bound(g.offsets, g.src, iters=8, resid=wres)
        check_pagerank(rank[bp.vbase[i]:bp.vbase[i + 1]], want, bound, 1e-5, what=f"graph {i}")
        assert np.all(np.abs(res[i] - wres) <= 1e-2 * wres + 2.4e-7), i


def test_sources_outside_their_graph_are_left_out():
    import torch
    from paper_1608_01362_gb300 import cagra as C
    off = np.array([0, 3, 5, 6, 6], np.int64)  # graphs of 3 and 1 vertices
    src = np.array([0, 1, 77, 2, -5, 0], np.int32)
    keep = np.array([0, 1, 2, 0], np.int32)  # what is inside
    koff = np.array([0, 2, 3, 4, 4], np.int64)
    out = []
    for o, s in ((off, src), (koff, keep)):
        b = C.pr_batch_create([0, 3, 4], torch.as_tensor(o).cuda(), torch.as_tensor(s).cuda())
        r = torch.empty(4, dtype=torch.float32, device="cuda")
        C.pr_batch_run(b, 5, 0.85, r)
        out.append(r.cpu().numpy())
    assert np.allclose(out[0], out[1], rtol=1e-6, atol=0)
