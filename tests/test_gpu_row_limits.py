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


def test_relabel_of_more_than_2_31_edges():
    import torch
    from paper_1608_01362_gb300 import cagra as C
    n = [2 ** 30 + 7, 3, 0, 2 ** 30 + 1001, 40_000]
    V, E = len(n), sum(n)
    assert E > 2 ** 31
    off = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.tensor(n, device="cuda"), 0)
    src = torch.randint(0, V, (E,), dtype=torch.int32, device="cuda")
    n2o = torch.tensor([3, 0, 4, 1, 2], dtype=torch.int32, device="cuda")  # new ID of each old one
    o2n = torch.argsort(n2o).int()
    noff, nsrc = torch.empty_like(off), torch.empty_like(src)
    C.cg_relabel_csr(off, src, n2o, o2n, noff, nsrc)
    want = [n[o] for o in o2n.tolist()]
    assert (noff[1:] - noff[:-1]).tolist() == want
    for new, old in enumerate(o2n.tolist()):
        a, b = int(noff[new]), int(off[old])
        for i in range(0, n[old], 2 ** 28):
            m = min(2 ** 28, n[old] - i)
            assert torch.equal(nsrc[a + i:a + i + m], n2o[src[b + i:b + i + m]]), (new, i)


def test_relabel_with_a_repeated_row_stays_within_its_edges():
    """An old_of_new that is no permutation may ask for more edges than there are
    (here 20 hub rows of 2^27): those past the last are left out."""
    import torch
    from paper_1608_01362_gb300 import cagra as C
    V, hub = 24, 2 ** 27
    off = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
    off[6:] = hub  # row 5
    off[V] = hub + 2  # the last row: two edges
    src = torch.randint(0, V, (hub + 2,), dtype=torch.int32, device="cuda")
    ident = torch.arange(V, dtype=torch.int32, device="cuda")
    o2n = torch.full((V,), 5, dtype=torch.int32, device="cuda")
    o2n[0] = V - 1
    noff, nsrc = torch.empty_like(off), torch.empty_like(src)
    C.cg_relabel_csr(off, src, ident, o2n, noff, nsrc)
    assert int(noff[V]) == 2 + (V - 1) * hub
    assert torch.equal(nsrc, torch.cat([src[hub:], src[:hub]]))
