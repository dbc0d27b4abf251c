"""Betweenness where its tiles meet their edges: rows over many gather tiles, the
long tiles of large levels, levels of one vertex, sources whose graph is all
push or all pull.  Levels and path counts bit for bit; dependencies within
2 * depth * (max degree + 8) * 2^-53 of the oracle (every term is positive, each
level adds at most deg + 3 roundings on either side)."""
import numpy as np
import pytest

import graphgen
import oracle as O

pytestmark = pytest.mark.gpu


def _graph(name):
    if name == "hubs":  # two vertices with 20,000 in- and out-edges each, among short rows
        rng = np.random.default_rng(4)
        n = 30_000
        a = rng.choice(n, 20_000, replace=False)
        b = rng.choice(n, 20_000, replace=False)
        s = np.concatenate([a, np.zeros(20_000, int), b, np.ones(20_000, int),
                            rng.integers(0, n, 40_000)])
        d = np.concatenate([np.zeros(20_000, int), b, np.ones(20_000, int), a,
                            rng.integers(0, n, 40_000)])
        return graphgen.from_edges(n, s, d)
    if name == "layers":  # levels of 1, 256, 257, 1 and 3000 vertices, fully joined
        sizes = [1, 256, 257, 1, 3000]
        at = np.concatenate([[0], np.cumsum(sizes)])
        s, d = [], []
        for i in range(len(sizes) - 1):
            p, q = np.arange(at[i], at[i + 1]), np.arange(at[i + 1], at[i + 2])
            s.append(np.repeat(p, len(q)))
            d.append(np.tile(q, len(p)))
        return graphgen.from_edges(int(at[-1]) + 9, np.concatenate(s), np.concatenate(d))
    return graphgen.rmat(19, 20, seed=6)  # levels of more than 2^22 edges


@pytest.mark.parametrize("alpha", [0.0, 16.0, 1e12])
@pytest.mark.parametrize("name", ["hubs", "layers", "rmat19"])
def test_levels_counts_dependencies(name, alpha):
    import torch
    from paper_1608_01362_gb300 import pipeline as P
    g = _graph(name)
    oo, od = O.out_csr(g.offsets, g.src)
    deg = int(np.diff(oo).max())
    for clustered in ((None,) if name == "rmat19" else (None, 0)):
        bc = P.Betweenness(P.Graph(g.offsets, g.src, cluster_mode=clustered), alpha=alpha)
        for s in [0, int(np.argmax(np.diff(oo)))]:
            lev, sig, delta = O.bc_source(oo, od, s)[:3]
            got = bc.run([s]).cpu().numpy()
            l, c, d, info = bc.source_state()
            assert np.array_equal(l.cpu().numpy(), lev)
            assert np.array_equal(c.cpu().numpy(), sig)
            assert info["depth"] == lev.max() + 1
            if alpha == 0.0:
                assert info["pull_levels"] == 0
            if alpha == 1e12:
                assert info["push_levels"] == 0
            tol = 2.0 * info["depth"] * (deg + 8) * 2.0 ** -53
            want = delta.copy()
            want[s] = 0.0
            assert np.all(np.abs(got - want) <= tol * np.abs(want))
            assert np.all(np.abs(d.cpu().numpy() - delta) <= tol * np.abs(delta))
            again = bc.run([s]).cpu().numpy()
            assert np.array_equal(again, got)
