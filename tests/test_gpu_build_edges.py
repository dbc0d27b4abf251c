"""Building the segmented structure where its passes can go wrong: edge counts
around the tiles, long runs of empty rows, hub rows over many tiles, segments
that begin inside a warp's edges, rows over many chunks.  Bit-exact against the
oracle (sums of small integers are exact in any order)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_1608_01362_gb300 import cagra
    return cagra


def _csr(name):
    rng = np.random.default_rng(7)
    if name.startswith("E"):  # E edges on rows of 0..3 edges
        E, V = int(name[1:]), 5000
        deg = np.bincount(rng.integers(0, V, E), minlength=V)
    elif name == "empties":  # a few rows between thousands of empty ones
        V = 200_000
        deg = np.zeros(V, np.int64)
        deg[rng.choice(V, 40, replace=False)] = rng.integers(1, 3000, 40)
        deg[0], deg[V - 1] = 5, 7
    elif name == "hub":  # one row of 300,000 edges (duplicates allowed) among short ones
        V = 3000
        deg = rng.integers(0, 3, V)
        deg[1234] = 300_000
    elif name == "last":  # every edge in the last row
        V = 4097
        deg = np.zeros(V, np.int64)
        deg[-1] = 2049
    off = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    return off, rng.integers(0, V, off[-1]).astype(np.int32)


NAMES = ["E1", "E31", "E2047", "E2048", "E2049", "E4096", "E30011", "empties", "hub", "last"]


@pytest.mark.parametrize("k", [1, 2, 33, 1000])
@pytest.mark.parametrize("name", NAMES)
def test_segments_and_sums(C, name, k):
    import torch
    off, src = _csr(name)
    V = len(off) - 1
    d_off, d_src = torch.as_tensor(off).cuda(), torch.as_tensor(src).cuda()
    ref = O.build_segments(off, src, k=k, B=512)
    seg = C.pr_build_segments(d_off, d_src, k)
    got = C.cg_segmented_export(seg)
    for f in ("bounds", "row_base", "edge_base", "row_ptr", "col", "idx_map", "block_start"):
        assert np.array_equal(got[f], getattr(ref, f)), f
    # all segments through L1/L2, so that the hub's row runs over many chunks
    C.pr_set_gather_config(seg, 1024, 1, 0)
    lab = np.random.default_rng(1).permutation(V).astype(np.int32)
    want = np.minimum.reduceat(lab[ref.col], ref.row_ptr[:-1])
    ones = np.ones(V, np.float32)
    for _ in range(2):
        g = torch.full((ref.rows,), -7, dtype=torch.int32, device="cuda")
        C.cg_seg_gather(seg, C.CG_OP_MIN_I32, torch.as_tensor(lab).cuda(), g)
        assert np.array_equal(g.cpu().numpy(), want)
        f = torch.full((ref.rows,), -1.0, device="cuda")
        C.cg_seg_gather(seg, C.CG_OP_SUM_F32, torch.as_tensor(ones).cuda(), f)
        assert np.array_equal(f.cpu().numpy().astype(np.int64), np.diff(ref.row_ptr))


@pytest.mark.parametrize("name", NAMES)
def test_relabel(C, name):
    import torch
    off, src = _csr(name)
    V = len(off) - 1
    n2o = np.random.default_rng(9).permutation(V).astype(np.int32)
    o2n = np.empty_like(n2o)
    o2n[n2o] = np.arange(V, dtype=np.int32)
    want_off, want_src = O.relabel(off, src, n2o, o2n)
    d = [torch.as_tensor(a).cuda() for a in (off, src, n2o, o2n)]
    noff, nsrc = torch.empty_like(d[0]), torch.empty_like(d[1])
    C.cg_relabel_csr(*d, noff, nsrc)
    assert np.array_equal(noff.cpu().numpy(), want_off)
    assert np.array_equal(nsrc.cpu().numpy(), want_src)


@pytest.mark.parametrize("V", [1, 31, 1000, 70_001])
@pytest.mark.parametrize("smem", [0, 1, 33, 512])
def test_plan_bounds(C, V, smem):
    import torch
    rng = np.random.default_rng(V)
    deg = np.sort(rng.integers(0, 40, V))[::-1].astype(np.int32).copy()
    for tail in (0, V // 3, V):
        deg[V - tail:] = 0
        got = C.pr_plan_bounds(torch.as_tensor(deg).cuda(), smem, 10.0, 5000, 64)
        b, lo = [0], 0  # the rule, restated on the host
        while smem > 0 and lo < V and len(b) < 64:
            n = min(smem, V - lo)
            if deg[lo:lo + n].sum() < 10.0 * n:
                break
            lo += n
            b.append(lo)
        if lo < V:
            nz = np.flatnonzero(deg)
            end = max(lo, int(nz[-1]) + 1 if len(nz) else 0)
            left = 64 - (len(b) - 1) - (1 if end < V and end > lo else 0)
            if left < 1:
                b[-1] = V
            else:
                if end > lo:
                    parts = min(max(1, -(-(end - lo) // 5000)), left)
                    step = -(-(end - lo) // parts)
                    b += [min(end, lo + q * step) for q in range(1, parts + 1)]
                if b[-1] < V:
                    b.append(V)
        assert got.tolist() == b, (tail, got, b)
