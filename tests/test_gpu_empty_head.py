"""The overlapped gather on plans whose leading staged segments are all empty:
there are no staged tasks, so it stays off, and the sums are those of two
launches; freshly built, and after a shape that staged more."""
import numpy as np
import pytest

import graphgen
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bounds,table", [((0, 0, 4096), 64), ((0, 0, 0, 3000, 4096), 64),
                                          ((0, 0, 4096), 0), ((0, 0, 2048, 4096), -1)])
def test_overlap_needs_staged_tasks(bounds, table):
    import torch
    from paper_1608_01362_gb300 import cagra as C
    g = graphgen.rmat(12, 12, seed=3)
    b = np.asarray(bounds, np.int64)
    ref = O.build_segments(g.offsets, g.src, k=len(b) - 1, B=512, bounds=b)
    seg = C.pr_build_segments(torch.as_tensor(g.offsets).cuda(), torch.as_tensor(g.src).cuda(),
                              len(b) - 1, bounds=b)  # the other segments are staged at first
    lab = np.random.default_rng(1).permutation(g.V).astype(np.int32)
    want = np.minimum.reduceat(lab[ref.col], ref.row_ptr[:-1])
    x = torch.rand(g.V, generator=torch.Generator().manual_seed(2)).cuda()

    def sums():
        f = torch.full((ref.rows,), -1.0, device="cuda")
        m = torch.full((ref.rows,), -7, dtype=torch.int32, device="cuda")
        C.cg_seg_gather(seg, C.CG_OP_SUM_F32, x, f)
        C.cg_seg_gather(seg, C.CG_OP_MIN_I32, torch.as_tensor(lab).cuda(), m)
        return f, m

    C.pr_set_gather_config(seg, 1024, 1, table)
    before = sums()
    assert np.array_equal(before[1].cpu().numpy(), want)
    C.pr_set_gather_overlap(seg, 8)
    info = seg.info
    staged = info["staged_edges"] > 0 and info["staged_edges"] < g.E
    assert info["gather_overlap"] == (8 if staged else 0)  # before any launch
    after = sums()
    assert torch.equal(after[0], before[0]) and torch.equal(after[1], before[1])
