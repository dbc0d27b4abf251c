"""The merge's own block size (the caller's, or one that makes whole waves of warps)
and the counters that a launch leaves cleared for the next one: exact against
numpy, over sizes at the edges of a block and over every way to run a gather."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_1608_01362_gb300 import cagra
    return cagra


def _graph(V, E, seed):
    rng = np.random.default_rng(seed)
    dst = np.sort((V * rng.random(E) ** 2).astype(np.int64))
    src = (V * rng.random(E) ** 3).astype(np.int64)
    keep = np.unique(dst * V + src)
    dst, src = keep // V, keep % V
    off = np.zeros(V + 1, np.int64)
    np.cumsum(np.bincount(dst, minlength=V), out=off[1:])
    return off, src.astype(np.int32), dst


@pytest.mark.parametrize("V", [1, 31, 33, 511, 4097, 70_001, 500_003])
@pytest.mark.parametrize("B", [1, 33, 511, 6144])
def test_sums_and_minima(C, V, B):
    import torch
    off, src, dst = _graph(V, max(1, 4 * V), V + B)
    seg = C.pr_build_segments(torch.as_tensor(off).cuda(), torch.as_tensor(src).cuda(),
                              min(3, V), merge_block=B)
    info = seg.info
    assert info["merge_block"] == B and info["num_blocks"] == -(-V // B)
    x = (1 + np.arange(V) % 5).astype(np.float32)
    lab = np.random.default_rng(2).permutation(V).astype(np.int32)
    sums = np.bincount(dst, weights=x[src], minlength=V).astype(np.float32)
    low = np.full(V, np.iinfo(np.int32).max, np.int32)
    np.minimum.at(low, dst, lab[src])
    for op, vec, want in ((C.CG_OP_SUM_F32, x, sums), (C.CG_OP_MIN_I32, lab, low)):
        d = torch.as_tensor(vec).cuda()
        interm = torch.zeros(max(1, info["rows"]), dtype=d.dtype, device="cuda")
        C.cg_seg_gather(seg, op, d, interm)
        out = torch.empty_like(d)
        C.merge(seg, op, interm, out)
        assert np.array_equal(out.cpu().numpy(), want)


def test_counters_are_left_cleared(C):
    """One plan, every kind of launch after every other: each run's result is
    the first one's."""
    import torch
    V = 200_003
    off, src, dst = _graph(V, 3_000_000, 7)
    seg = C.pr_build_segments(torch.as_tensor(off).cuda(), torch.as_tensor(src).cuda(), 24)
    x = (1 + np.arange(V) % 3).astype(np.float32)
    want = np.bincount(dst, weights=x[src], minlength=V).astype(np.float32)
    d = torch.as_tensor(x).cuda()
    interm = torch.zeros(seg.info["rows"], dtype=torch.float32, device="cuda")
    out = torch.empty_like(d)
    rng = np.random.default_rng(1)
    for _ in range(6):
        for how in rng.permutation(4):
            C.pr_set_gather_overlap(seg, 0)
            C.pr_set_gather_affine(seg, 0.0)
            C.pr_set_gather_config(seg, *((512, 2) if how == 1 else (1024, 1)))
            if how == 2:
                C.pr_set_gather_overlap(seg, 8)
            if how == 3:
                C.pr_set_gather_affine(seg, 5.0)
            for _ in range(2):
                C.cg_seg_gather(seg, C.CG_OP_SUM_F32, d, interm)
                C.merge(seg, C.CG_OP_SUM_F32, interm, out)
                assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("V", [1, 255, 256, 257, 1_000_001])
def test_start_counts_its_dangling_mass(C, V):
    import torch
    inv = (np.arange(V) % 3).astype(np.float32)
    D = torch.full((1,), 7.0, dtype=torch.float64, device="cuda")
    rank, contrib = (torch.empty(V, dtype=torch.float32, device="cuda") for _ in range(2))
    d = torch.as_tensor(inv).cuda()
    for _ in range(2):
        C.pr_init(d, rank, contrib, D)
        r = np.float32(1) / np.float32(V)
        assert D.item() == float((V + 2) // 3) * float(r)
        assert np.array_equal(rank.cpu().numpy(), np.full(V, r))
        assert np.array_equal(contrib.cpu().numpy(), r * inv)


@pytest.mark.parametrize("drop", [0, 1])
def test_chunks_of_the_cached_segments(C, drop):
    """2^24 edges read through L1/L2, and one fewer: the two chunk sizes."""
    import torch
    V = 1 << 20
    src = (np.arange(16) * 65536 + (np.arange(V) * 7919 % 65536)[:, None]).astype(np.int32).ravel()
    src = src[:src.size - drop]
    off = np.minimum(np.arange(V + 1, dtype=np.int64) * 16, src.size)
    seg = C.pr_build_segments(torch.as_tensor(off).cuda(), torch.as_tensor(src).cuda(), 1)
    assert seg.info["staged_segments"] == 0
    x = (1 + np.arange(V) % 7).astype(np.float32)
    want = np.add.reduceat(x[src], off[:-1])
    out = torch.full((V,), -1.0, device="cuda")
    for _ in range(2):
        C.cg_seg_gather(seg, C.CG_OP_SUM_F32, torch.as_tensor(x).cuda(), out)
        assert np.array_equal(out.cpu().numpy(), want)
