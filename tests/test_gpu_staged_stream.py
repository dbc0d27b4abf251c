"""The staged segments' stream: rows at the edges of its length classes, of its
windows and of its full pieces, exact against numpy (integer sums below 2^24
and minima do not depend on the order)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    from paper_1608_01362_gb300 import cagra
    return cagra


EDGES = [1, 2, 3, 4, 5, 6, 7, 8, 9, 15, 16, 17, 18, 31, 32, 33, 63, 64, 65, 128, 129, 256, 257, 511,
         512, 513, 767, 768, 769, 1024, 1025, 4095, 4096, 4097, 4608, 8191, 8192, 8193, 9000]


def _rows(lengths, V):
    rng = np.random.default_rng(5)
    src = [np.sort(rng.choice(V, n, replace=False)) for n in lengths]
    off = np.zeros(V + 1, np.int64)
    off[1:len(lengths) + 1] = np.cumsum(lengths)
    off[len(lengths) + 1:] = off[len(lengths)]
    return off, np.concatenate(src).astype(np.int32)


def _cases():
    rng = np.random.default_rng(3)
    return {
        "class_edges": (rng.permutation(np.repeat(EDGES, 3)), 9001),
        "one_row": (np.array([9000]), 2000 + 7001),
        "short": (rng.integers(1, 4, 8999), 4001 + 5000),
        # more rows than a window holds, most of one class
        "windows": (np.where(np.arange(70_000) % 1000 == 0, 513, rng.integers(1, 18, 70_000)),
                    70_001),
    }


@pytest.mark.parametrize("name", list(_cases()))
@pytest.mark.parametrize("shape", [(1024, 1), (512, 2)])
@pytest.mark.parametrize("k", [1, 3])
def test_rows_of_every_class(C, name, shape, k):
    import torch
    lengths, V = _cases()[name]
    off, src = _rows(lengths, V)
    # leading segments dense enough to be staged
    if k == 1 and V > 25_000:
        bounds = np.array([0, 25_000, V])
    else:
        bounds = np.linspace(0, V, k + 1).astype(np.int64)
    seg = C.pr_build_segments(torch.as_tensor(off).cuda(), torch.as_tensor(src).cuda(),
                              len(bounds) - 1, bounds=bounds)
    C.pr_set_gather_config(seg, *shape)
    info = seg.info
    if name in ("class_edges", "windows"):
        assert info["staged_segments"] >= 1
    x = (1 + np.arange(V) * 2654435761 % 5).astype(np.float32)
    lab = np.random.default_rng(2).permutation(V).astype(np.int32)
    ex = C.cg_segmented_export(seg)
    rp = ex["row_ptr"][:-1]
    want = np.add.reduceat(x[ex["col"]].astype(np.int64), rp)
    wmin = np.minimum.reduceat(lab[ex["col"]], rp)
    got = torch.full((info["rows"],), float("nan"), device="cuda")
    gmin = torch.full((info["rows"],), -7, dtype=torch.int32, device="cuda")
    xd, ld = torch.as_tensor(x).cuda(), torch.as_tensor(lab).cuda()
    for affine in ([0.0, 5.0] if shape == (1024, 1) else [0.0]):
        if shape == (1024, 1):
            C.pr_set_gather_affine(seg, affine)
        for _ in range(2):  # the launch leaves its counters ready for the next
            got.fill_(float("nan"))
            gmin.fill_(-7)
            C.cg_seg_gather(seg, C.CG_OP_SUM_F32, xd, got)
            C.cg_seg_gather(seg, C.CG_OP_MIN_I32, ld, gmin)
            assert np.array_equal(got.cpu().numpy().astype(np.int64), want)
            assert np.array_equal(gmin.cpu().numpy(), wmin)
    # infinities and NaN stay in the rows that read them
    xi = x.copy()
    xi[src[0]], xi[src[-1]] = np.inf, np.nan
    C.cg_seg_gather(seg, C.CG_OP_SUM_F32, torch.as_tensor(xi).cuda(), got)
    with np.errstate(invalid="ignore"):
        wi = np.add.reduceat(xi[ex["col"]].astype(np.float64), rp)
    g = got.cpu().numpy().astype(np.float64)
    assert np.array_equal(np.isnan(g), np.isnan(wi))
    assert np.array_equal(np.isinf(g), np.isinf(wi))
    assert np.array_equal(g[np.isfinite(wi)], wi[np.isfinite(wi)])
