"""Betweenness from several threads at once, each with a handle and a stream of
its own: the level counts that a run reads from its pinned words are its own.
Dependencies within 2 * depth * (max degree + 8) * 2^-53 of each other (every
term is positive, each level adds at most deg + 3 roundings on either side),
depth below 64 here."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _graph(torch, P, V, seed):
    rng = np.random.default_rng(seed)
    key = np.unique(rng.integers(0, V, 6 * V) * V + (V * rng.random(6 * V) ** 2).astype(np.int64))
    off = np.zeros(V + 1, np.int64)
    np.cumsum(np.bincount(key // V, minlength=V), out=off[1:])
    return P.Graph(torch.as_tensor(off).cuda(), torch.as_tensor((key % V).astype(np.int32)).cuda(),
                   cluster_mode=None)


@pytest.mark.parametrize("sizes", [(1, 40, 3000, 60_000)])
def test_runs_side_by_side(sizes):
    import torch
    from paper_1608_01362_gb300 import pipeline as P
    graphs = [_graph(torch, P, V, V) for V in sizes]
    sources = [[(7 * q) % V for q in range(5)] for V in sizes]
    alone = [P.Betweenness(g).run(s).clone() for g, s in zip(graphs, sources)]
    torch.cuda.synchronize()
    got, failed = [None] * len(sizes), []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                b = P.Betweenness(graphs[i])
                for _ in range(8):
                    got[i] = b.run(sources[i]).clone()
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # reported by the main thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for g, a, b in zip(graphs, alone, got):
        deg = int(torch.bincount(g.src, minlength=1).max()) if g.E else 0
        assert torch.allclose(a, b, rtol=2 * 64 * (deg + 8) * 2.0 ** -53, atol=0)
