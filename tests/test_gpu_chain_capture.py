"""Chained launches (each waits at its start for the one before) captured in a
CUDA graph and replayed: the results are those of the plain calls."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1608_01362_gb300 import cagra as C, pipeline as P
    g = graphgen.rmat(15, 16, seed=3)
    return torch, C, P, P.Graph(g.offsets, g.src, cluster_mode=0)


def _replayed(torch, call):
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        call()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()


@pytest.mark.parametrize("k", [1, 5])
def test_pagerank(env, k):
    torch, C, P, g = env
    pr = P.SegmentedPageRank(g, k)
    want = pr.run(7)[0].clone()
    out, contrib = torch.empty_like(pr.rank[0]), torch.empty_like(pr.contrib[0])

    def call():
        pr.init()
        C.pr_iterate(pr.seg, g.inv, pr.rank[0], pr.contrib[0], out, contrib, 0.85, 7, pr.dangling,
                     None)
    _replayed(torch, call)
    assert torch.equal(g.to_original(out), want)


def test_batched_ppr(env):
    torch, C, P, g = env
    b = P.BatchedPPR(g, 2)
    seeds = (np.arange(64) * 31) % g.V
    want = b.run(seeds, iterations=9)[0].clone()
    out = torch.empty_like(b.rank)
    b.init(seeds)
    one = lambda: C.ppr_batched_iterate(b.ppr, g.inv, 0.85, 3, out, None)  # noqa: E731
    _replayed(torch, one)  # three replays of three iterations
    assert torch.equal(g.rows_to_original(out), want)


def test_collaborative_filtering(env):
    torch, C, P, _ = env
    rng = np.random.default_rng(1)
    U, I, K = 700, 300, 32
    rows = [np.sort(rng.choice(I, int(n), replace=False)) for n in rng.integers(0, 90, U)]
    off = torch.as_tensor(np.concatenate([[0], np.cumsum([len(r) for r in rows])])).cuda()
    item = torch.as_tensor(np.concatenate(rows).astype(np.int32)).cuda()
    rate = torch.as_tensor(rng.integers(1, 6, item.numel()).astype(np.uint8)).cuda()
    ioff = torch.empty(I + 1, dtype=torch.int64, device="cuda")
    iuser, irate = torch.empty_like(item), torch.empty_like(rate)
    C.cf_transpose(U, I, off, item, rate, ioff, iuser, irate)
    h = C.cf_create(U, I, K, 0, off, item, rate, ioff, iuser, irate)
    P0 = torch.as_tensor(rng.random((U, K)).astype(np.float32)).cuda()
    Q0 = torch.as_tensor(rng.random((I, K)).astype(np.float32)).cuda()
    sse = torch.zeros(3, dtype=torch.float64, device="cuda")
    got = [torch.empty_like(P0), torch.empty_like(Q0)]
    C.cf_set_factors(h, P0, Q0)
    C.cf_sweep(h, 9, 0.05, 1e-3, None)
    C.cf_get_factors(h, *got)
    want = [x.clone() for x in got]
    C.cf_set_factors(h, P0, Q0)
    _replayed(torch, lambda: C.cf_sweep(h, 3, 0.05, 1e-3, sse))
    C.cf_get_factors(h, *got)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
