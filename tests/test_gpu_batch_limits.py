"""Batches beyond what one launch takes: more than 2^18 graphs, more than 2^31 edges
in total.  Copies of one graph have the ranks that it has alone, bit for bit."""
import numpy as np
import pytest

import graphgen
import oracle as O
from parity import check_pagerank

pytestmark = pytest.mark.gpu


def _copies(torch, g, n):
    """n copies of graph g, end to end, made on the GPU."""
    off = torch.as_tensor(g.offsets[:-1]).cuda()
    offsets = torch.empty(n * g.V + 1, dtype=torch.int64, device="cuda")
    offsets[:-1] = (off[None, :] + (torch.arange(n, device="cuda") * g.E)[:, None]).flatten()
    offsets[-1] = n * g.E
    return np.arange(n + 1, dtype=np.int64) * g.V, offsets, torch.as_tensor(g.src).cuda().repeat(n)


def _run(torch, C, vbase, offsets, src, resid=None):
    rank = torch.empty(int(vbase[-1]), dtype=torch.float32, device="cuda")
    C.pr_batch_run(C.pr_batch_create(vbase, offsets, src), 6, 0.85, rank, resid)
    return rank


@pytest.mark.parametrize("n,scale,factor", [(2 ** 18 + 37, 5, 3), (4200, 15, 18)])
def test_copies(n, scale, factor):
    import torch
    from paper_1608_01362_gb300 import cagra as C
    g = graphgen.rmat(scale, factor, seed=6)
    assert n > 2 ** 18 or n * g.E > 2 ** 31
    one = _run(torch, C, np.array([0, g.V]), torch.as_tensor(g.offsets).cuda(),
               torch.as_tensor(g.src).cuda())
    want, bound = O.pagerank_bound(g.offsets, g.src, iters=6)
    check_pagerank(one.cpu().numpy(), want, bound)
    resid = torch.full((n * 6,), -1.0, dtype=torch.float64, device="cuda")
    got = _run(torch, C, *_copies(torch, g, n), resid).view(n, g.V)
    assert torch.equal(got, one[None, :].expand(n, g.V))
    assert torch.equal(resid.view(n, 6), resid[:6][None, :].expand(n, 6)) and bool(resid[0] > 0)


def test_graphs_of_different_sizes_over_the_border():
    import torch
    from paper_1608_01362_gb300 import cagra as C, pipeline as P
    n = 2 ** 18 - 2  # the last graphs lie on both sides of the first part's end
    tiny = graphgen.from_edges(3, [0, 1, 1], [1, 2, 0])
    rest = [graphgen.rmat(s, 5, seed=s) for s in (9, 6, 11, 3, 8)]
    vb, off, src = _copies(torch, tiny, n)
    rvb, roff, rsrc = P.concat_graphs(rest)
    vbase = np.concatenate([vb, rvb[1:] + vb[-1]])
    offsets = torch.cat([off[:-1], torch.as_tensor(roff).cuda() + n * tiny.E])
    rank = _run(torch, C, vbase, offsets, torch.cat([src, torch.as_tensor(rsrc).cuda()]))
    rank = rank[n * 3:].cpu().numpy()
    for i, g in enumerate(rest):
        want, bound = O.pagerank_bound(g.offsets, g.src, iters=6)
        check_pagerank(rank[rvb[i]:rvb[i + 1]], want, bound, what=f"graph {i}")
