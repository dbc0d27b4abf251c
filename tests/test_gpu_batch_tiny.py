"""Thousands of tiny graphs in a batch: each has the ranks and residuals, bit for
bit, that it has alone, around the row lengths where the order of a sum changes and
the sizes up to which a graph is tiny; and they take little more memory than their
edges."""
import numpy as np
import pytest

import graphgen
import oracle as O
from parity import check_pagerank

pytestmark = pytest.mark.gpu
ROWS = [0, 1, 2, 3, 4, 5, 7, 8, 9, 10, 15, 16, 17, 31, 32, 33, 63, 64, 65, 100, 128, 129, 255]


class _Csr:
    def __init__(self, V, lengths, rng, outside=False):
        self.V = V
        self.offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
        self.src = rng.integers(0, V, self.offsets[-1]).astype(np.int32)  # some edges repeat
        if outside:
            self.src[::5] = V + rng.integers(0, 300, self.src[::5].size)
            self.src[3::11] = -1 - rng.integers(0, 300, self.src[3::11].size)


def _graphs():
    rng = np.random.default_rng(11)
    out = [_Csr(n + 1, [n] + [0] * n, rng) for n in ROWS]  # one row of n edges
    for V in (1, 2, 31, 32, 33, 64, 65, 200, 255, 256):  # 255 vertices: the most
        out.append(_Csr(V, rng.integers(0, 9, V) * (rng.random(V) < 0.7), rng))
    for n in (1279, 1280, 1281):  # 1280 edges: the most
        out.append(_Csr(200, np.bincount(rng.integers(0, 200, n), minlength=200), rng))
    out.append(_Csr(90, np.bincount(rng.integers(0, 9, 300), minlength=90), rng, outside=True))
    out.append(_Csr(255, [256] + [1] * 254, rng))  # a row too long
    return out


@pytest.mark.parametrize("threads", [1024, 512, 256])
def test_as_alone(threads):
    import torch
    from paper_1608_01362_gb300 import pipeline as P
    gs, it = _graphs(), 7

    def run(graphs, resid):
        b = P.BatchedPageRank(graphs, threads=threads)
        r = torch.zeros(len(graphs) * it, dtype=torch.float64, device="cuda") if resid else None
        rank = b.run(it, resid=r).cpu().numpy()
        return b.vbase, rank, r.cpu().numpy().reshape(-1, it) if resid else None

    alone = []
    for g in gs:
        _, rank, res = run([g], True)
        alone.append((rank, res[0]))
        if np.all((g.src >= 0) & (g.src < g.V)):
            want, bound = O.pagerank_bound(g.offsets, g.src, iters=it)
            check_pagerank(rank, want, bound)
    many = gs * (5000 // len(gs))
    for resid in (True, False):
        vbase, rank, res = run(many, resid)
        for i in range(len(many)):
            r, q = alone[i % len(gs)]
            assert np.array_equal(rank[vbase[i]:vbase[i + 1]], r), i % len(gs)
            assert not resid or np.array_equal(res[i], q), i % len(gs)


def test_memory():
    import torch
    from paper_1608_01362_gb300 import cagra as C
    G, V, deg = 20_000, 25, 2
    off = torch.zeros(G * V + 1, dtype=torch.int64, device="cuda")  # rows of 0 to about 12
    row = torch.randint(0, G * V, (G * V * deg,), device="cuda")
    torch.cumsum(torch.bincount(row, minlength=G * V), 0, out=off[1:])
    src = torch.randint(0, V, (G * V * deg,), dtype=torch.int32, device="cuda")
    vbase = np.arange(G + 1, dtype=np.int64) * V
    C.pr_batch_create(vbase, off, src)  # what the library keeps from a first call
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    batch = C.pr_batch_create(vbase, off, src)
    torch.cuda.synchronize()
    kept = before - torch.cuda.mem_get_info()[0]
    # 16 bytes per vertex, 80 per graph, 1 per edge; allocations in steps of 2 MB
    assert kept <= 16 * G * V + 80 * G + G * V * deg + 16 * 2 ** 21, kept
    del batch
