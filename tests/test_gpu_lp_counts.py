"""Label propagation's counts of changed labels: those that a run takes from its
pinned words are those of single passes, whatever ran on the handle before."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 6])
@pytest.mark.parametrize("scale", [6, 13])
def test_run_counts_as_single_passes_do(scale, k):
    import torch
    from paper_1608_01362_gb300 import cagra as C, pipeline as P
    g = graphgen.rmat(scale, 8, seed=5, symmetric=True)
    seg = C.pr_build_segments(torch.as_tensor(g.offsets).cuda(), torch.as_tensor(g.src).cuda(), k)
    start = torch.arange(g.V, dtype=torch.int32, device="cuda")
    a, b, want = start.clone(), torch.empty_like(start), []
    while not want or want[-1]:
        want.append(C.lp_iterate(seg, a, b))
        a, b = b, a
    x = torch.ones(g.V, device="cuda")
    for _ in range(3):
        lab = start.clone()
        passes, changes = C.lp_run(seg, lab)
        assert passes == len(want) and np.array_equal(np.asarray(changes)[:passes], want)
        assert torch.equal(lab, a)
        passes, changes = C.lp_run(seg, start.clone(), max_passes=2)  # ends before the end
        assert passes == min(2, len(want)) and np.array_equal(changes[:passes], want[:passes])
        assert C.lp_iterate(seg, start, b) == want[0]
        C.cg_seg_gather(seg, C.CG_OP_SUM_F32, x)
        C.merge(seg, C.CG_OP_SUM_F32, torch.zeros(seg.info["rows"], device="cuda"),
                torch.empty_like(x))
