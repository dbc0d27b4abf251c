"""The row walk at the limits of its types: as many vertices as an int32 holds
(nearly all of them without edges), and more than 2^31 edges in a renumbering.
Exact."""
import pytest

pytestmark = pytest.mark.gpu
V31 = 2 ** 31 - 1


def _offsets(torch, V, rows):
    """Offsets of V rows of which the listed (row, edges) have any."""
    off = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
    for r, n in rows:
        off[r + 1:] += n
    return off


def test_transpose_of_the_most_vertices():
    import torch
    from paper_1608_01362_gb300 import cagra as C
    edges = [(0, 0), (0, 5), (0, V31 - 1), (7, 5), (V31 - 33, 9), (V31 - 2, 0), (V31 - 1, V31 - 1)]
    by_row = sorted({(d, sum(e[0] == d for e in edges)) for d, _ in edges})  # (destination, source)
    off = _offsets(torch, V31, by_row)
    src = torch.tensor([s for _, s in edges], dtype=torch.int32, device="cuda")
    out_off, out_dst = torch.empty_like(off), torch.empty_like(src)
    C.cg_transpose_csr(off, src, out_off, out_dst)
    back = sorted((s, d) for d, s in edges)
    assert out_dst.tolist() == [d for _, d in back]
    del off
    want = _offsets(torch, V31, sorted({(s, sum(e[0] == s for e in back)) for s, _ in back}))
    assert torch.equal(out_off, want)
