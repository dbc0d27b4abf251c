"""A launch shape that there is no memory for: an error, and the handle goes on with
the previous shape or refuses to gather; with memory again it takes any shape."""
import pytest

pytestmark = pytest.mark.gpu


def test_shape_without_memory():
    import torch
    from paper_1608_01362_gb300 import cagra as C
    V, deg = 50_000, 12_000  # one staged segment; unstaged it takes 28 MB of carries
    off = torch.arange(0, V * deg + 1, deg, device="cuda")
    src = torch.randint(0, V, (V * deg,), dtype=torch.int32, device="cuda")
    seg = C.pr_build_segments(off, src, 1)
    assert seg.info["staged_edges"] == V * deg
    x = torch.ones(V, device="cuda")
    x[::3] = 2.0
    out = torch.zeros(V, device="cuda")
    C.cg_seg_gather(seg, C.CG_OP_SUM_F32, x, out)
    want = out.clone()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = [torch.empty(torch.cuda.mem_get_info()[0] - (20 << 20), dtype=torch.uint8,
                        device="cuda")]
    assert torch.cuda.mem_get_info()[0] < 24 << 20
    with pytest.raises(C.CagraError):
        C.pr_set_gather_config(seg, 1024, 1, 0)
    out.zero_()
    try:
        C.cg_seg_gather(seg, C.CG_OP_SUM_F32, x, out)
        assert torch.equal(out, want)
    except C.CagraError as e:
        assert "configur" in str(e)
    torch.cuda.synchronize()
    fill.clear()
    torch.cuda.empty_cache()
    for table in (0, -1):
        C.pr_set_gather_config(seg, 1024, 1, table)
        out.zero_()
        C.cg_seg_gather(seg, C.CG_OP_SUM_F32, x, out)
        assert torch.equal(out, want), table  # sums of integers below 2^24: exact
