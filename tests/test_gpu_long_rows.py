"""Rows of up to millions of edges read through L1/L2: exact sums and minima where
their carries begin and end at every place relative to the tiles that stand for
them, and no slower than a graph of short rows by more than a factor of 3."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rows(name):
    c = 128  # edges per carry at these sizes
    return {
        "one": [2_000_000],
        "between": [3, 700_000, 1, 900_001, 2] * 2,
        "ends with a tile": [512 * c, 1, 256 * 4 * c - 1, 5],
        "aligned": [1024 * c] * 3 + [7],
        "one edge more": [513 * c + 1, 511 * c - 1, 1025 * c + 1, 1],
        "shifted": [c * 31 + 5, 600 * c, c * 33 - 5, 777 * c + 13, 64 * c, 1500 * c - 1],
    }[name]


@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("name", ["one", "between", "ends with a tile", "aligned",
                                  "one edge more", "shifted"])
def test_sums_and_minima(name, k):
    import torch
    from paper_1608_01362_gb300 import cagra as C
    import oracle as O
    rng = np.random.default_rng(4)
    V = 3000
    deg = np.zeros(V, np.int64)
    lengths = _rows(name)
    deg[np.sort(rng.choice(V, len(lengths), replace=False))] = lengths
    off = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    src = rng.integers(0, V, off[-1]).astype(np.int32)
    ref = O.build_segments(off, src, k=k, B=512)
    seg = C.pr_build_segments(torch.as_tensor(off).cuda(), torch.as_tensor(src).cuda(), k)
    x = rng.integers(1, 6, V).astype(np.float32)
    lab = rng.permutation(V).astype(np.int32)
    want = np.add.reduceat(x[ref.col].astype(np.int64), ref.row_ptr[:-1])
    assert want.max() < 2 ** 24
    wmin = np.minimum.reduceat(lab[ref.col], ref.row_ptr[:-1])
    for table in (0, -1, 0):  # through L1/L2, staged, and back
        C.pr_set_gather_config(seg, 1024, 1, table)
        f = torch.full((ref.rows,), -1.0, device="cuda")
        m = torch.full((ref.rows,), -7, dtype=torch.int32, device="cuda")
        C.cg_seg_gather(seg, C.CG_OP_SUM_F32, torch.as_tensor(x).cuda(), f)
        C.cg_seg_gather(seg, C.CG_OP_MIN_I32, torch.as_tensor(lab).cuda(), m)
        assert np.array_equal(f.cpu().numpy().astype(np.int64), want), table
        assert np.array_equal(m.cpu().numpy(), wmin), table


def test_a_star_takes_no_longer_than_short_rows():
    import torch
    from paper_1608_01362_gb300 import cagra as C
    V = 1_000_003
    ms = {}
    for name in ("cycles", "star"):
        n = torch.full((V,), 2, dtype=torch.int64, device="cuda")
        if name == "star":
            n.fill_(1)
            n[0] += V
        off = torch.zeros(V + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(n, 0, out=off[1:])
        src = (torch.arange(int(off[-1]), device="cuda") % V).int()
        seg = C.pr_build_segments(off, src, 1)
        x = torch.ones(V, device="cuda")
        out = torch.empty(V, device="cuda")
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        for rep in range(30):
            if rep == 10:
                a.record()
            C.cg_seg_gather(seg, C.CG_OP_SUM_F32, x, out)
        b.record()
        b.synchronize()
        ms[name] = a.elapsed_time(b) / 20
        assert torch.equal(out, n.float())
    assert ms["star"] <= 3 * ms["cycles"], ms
