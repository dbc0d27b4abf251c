"""Batched personalised PageRank at the edges of its tasks, chunks and pieces
(destinations per octet, edges per chunk, chunks per piece): one iteration
exactly (each sum has one term that is not zero), three against FP64.

Three: every term is non-negative, so errors are relative, entry by entry.  A sum goes
through at most 128 edges, 16 chunks, the pieces of a row (< 64 here) and k
rows, each an FP32 rounding (2^-24): below 250 * 2^-24 = 1.5e-5 per iteration,
with the update's few roundings below 1.6e-5.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 3 * 1.6e-5
SIZES = [1, 15, 16, 17, 32, 33, 64, 127, 4097, 60_000]


def _graph(V):
    """Row 0 is read from everywhere, the others hold 0 to 300 edges."""
    rng = np.random.default_rng(V)
    n = np.minimum(rng.choice([0, 0, 1, 2, 3, 4, 5, 7, 8, 127, 128, 129, 300], V), V)
    n[0] = V
    n[V // 2] = min(V, 128 * 16)
    if V > 40_000:
        n[1:40_000] = np.minimum(n[1:40_000], 8)
    src = [np.sort(rng.choice(V, k, replace=False)) for k in n]
    off = np.zeros(V + 1, np.int64)
    np.cumsum(n, out=off[1:])
    return off, np.concatenate(src).astype(np.int32)


@pytest.mark.parametrize("V", SIZES)
@pytest.mark.parametrize("planes", [2, 1])
@pytest.mark.parametrize("k", [1, 3])
def test_one_iteration_is_exact(V, planes, k):
    import torch
    from paper_1608_01362_gb300 import pipeline as P
    off, src = _graph(V)
    graph = P.Graph(torch.as_tensor(off).cuda(), torch.as_tensor(src).cuda(), cluster_mode=None)
    seeds = (np.arange(64) * 977) % V
    c = graph.inv.cpu()
    c = (c if planes == 2 else c.to(torch.bfloat16).float()).numpy()[seeds]
    dst = np.repeat(np.arange(V), np.diff(off))
    want = np.zeros((V, 64), np.float32)
    for j, s in enumerate(seeds):
        want[dst[src == s], j] = np.float32(0.5) * c[j]
        want[s, j] += np.float32(0.5 if c[j] else 1.0)
    b = P.BatchedPPR(graph, min(k, V), planes=planes)
    for _ in range(2):
        assert np.array_equal(b.run(seeds, iterations=1, damping=0.5)[0].cpu().numpy(), want)


@pytest.mark.parametrize("V", SIZES)
@pytest.mark.parametrize("k", [1, 3])
def test_three_iterations(V, k):
    import torch
    from paper_1608_01362_gb300 import pipeline as P
    off, src = _graph(V)
    deg = np.bincount(src, minlength=V)
    inv = np.where(deg > 0, 1.0 / np.maximum(deg, 1), 0.0)
    dst = np.repeat(np.arange(V), np.diff(off))
    seeds = (np.arange(64) * 977) % V
    seeds[1] = 0
    d, R = 0.85, np.zeros((V, 64))
    R[seeds, np.arange(64)] = 1.0
    for _ in range(3):
        prev, C = R, R * inv[:, None]
        R = np.stack([np.bincount(dst, weights=C[src, j], minlength=V) for j in range(64)], 1) * d
        R[seeds, np.arange(64)] += (1 - d) + d * prev[deg == 0].sum(0)
    graph = P.Graph(torch.as_tensor(off).cuda(), torch.as_tensor(src).cuda(), cluster_mode=None)
    b = P.BatchedPPR(graph, min(k, V), planes=2)
    for _ in range(2):  # the counters are left ready
        got, resid = b.run(seeds, iterations=3, damping=d)
        got = got.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(got - R) <= TOL * R), np.max(np.abs(got - R))
        want = np.abs(R - prev).sum(0)
        assert np.allclose(resid.cpu().numpy(), want, rtol=0, atol=2 * TOL * 1.0001)
    # an output of the caller's that is only 16-byte aligned
    from paper_1608_01362_gb300 import cagra as C
    flat = torch.full((V * 64 + 8,), -1.0, device="cuda")
    out = flat[4:4 + V * 64].view(V, 64)
    b.init(seeds)
    C.ppr_batched_iterate(b.ppr, graph.inv, d, 3, out, None)
    assert np.array_equal(out.cpu().numpy().astype(np.float64), got)
    assert torch.all(flat[:4] == -1) and torch.all(flat[4 + V * 64:] == -1)
