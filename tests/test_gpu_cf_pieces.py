"""The collaborative-filtering gather where its pieces and tasks meet their edges:
rows of 15 to 33 ratings (pieces of 16 here), rows at the numbers of pieces from
which a warp (8) or a block (64) updates a vertex, vertices without ratings,
neighbours that ascend or not, every K and precision, ratings of 0 and 255.
Every entry within the oracle's rounding bound for a sweep from the same
factors (oracle.cf_sweep_bound: any summation tree)."""
import numpy as np
import pytest

import graphgen
import oracle as O

pytestmark = pytest.mark.gpu
LAM, STEP = 0.05, 1e-3


@pytest.fixture(scope="module")
def C():
    from paper_1608_01362_gb300 import cagra
    return cagra


@pytest.fixture(scope="module")
def ratings():
    rng = np.random.default_rng(8)
    U, I = 9001, 4503
    rows = []
    for u in range(U):
        if u % 97 == 0:
            rows.append(np.empty(0, np.int64))  # no ratings
        elif u < 160:
            n = [15, 16, 17, 31, 33, 128, 129, 1024, 1025, 4000][u % 10]
            rows.append(np.sort(rng.choice(I - 100, n, replace=False)))
        else:  # items rated by about 6,100 and by 300 to 500 users among them
            pick = np.unique((I * rng.random(40) ** 1.5).astype(np.int64))
            few = 4450 + np.flatnonzero(rng.random(40) < 0.045)
            rows.append(np.unique(np.concatenate([pick[pick < I - 110], few, [0] * (u < 6300)])))
    off = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    item = np.concatenate(rows).astype(np.int32)
    rate = rng.integers(0, 256, item.size).astype(np.uint8)
    return U, I, off, item, rate


def _item_major(C, U, I, off, item, rate):
    import torch
    d = [torch.as_tensor(a).cuda() for a in (off, item, rate)]
    ioff = torch.empty(I + 1, dtype=torch.int64, device="cuda")
    iuser, irate = torch.empty_like(d[1]), torch.empty_like(d[2])
    C.cf_transpose(U, I, *d, ioff, iuser, irate)
    return d + [ioff, iuser, irate]


@pytest.mark.parametrize("ascending", [True, False])
@pytest.mark.parametrize("K,precision", [(16, 0), (16, 1), (32, 0), (32, 1), (32, 2), (64, 0),
                                         (64, 2)])
def test_sweep_within_bound(C, ratings, K, precision, ascending):
    import torch
    U, I, off, item, rate = ratings
    u_store = {0: 0.0, 1: O.U_BF16, 2: O.U_BF16X2}[precision]
    d = _item_major(C, U, I, off, item, rate)
    if not ascending:  # every user's list turned round: the same ratings
        perm = np.concatenate([np.arange(a, b)[::-1] for a, b in zip(off[:-1], off[1:])])
        d[1] = torch.as_tensor(item[perm].copy()).cuda()
        d[2] = torch.as_tensor(rate[perm].copy()).cuda()
    h = C.cf_create(U, I, K, precision, *d)
    assert h.info["user_pieces"] == int(sum(-(-n // 16) for n in np.diff(off)))
    P0, Q0 = (0.05 * a for a in graphgen.cf_factors(U, I, K, seed=2))
    C.cf_set_factors(h, torch.as_tensor(P0.astype(np.float32)).cuda(),
                     torch.as_tensor(Q0.astype(np.float32)).cuda())
    Pg = torch.empty((U, K), dtype=torch.float32, device="cuda")
    Qg = torch.empty((I, K), dtype=torch.float32, device="cuda")
    sse = torch.zeros(1, dtype=torch.float64, device="cuda")
    ioff, iuser, irate = O.item_major(U, I, off, item, rate)
    for _ in range(2):
        C.cf_get_factors(h, Pg, Qg)
        P, Q = Pg.cpu().numpy().astype(np.float64), Qg.cpu().numpy().astype(np.float64)
        C.cf_sweep(h, 1, LAM, STEP, sse)
        C.cf_get_factors(h, Pg, Qg)
        Pn, Qn, s64, bP, bQ, bs = O.cf_sweep_bound(U, I, off, item, rate, ioff, iuser, irate, P, Q,
                                                   LAM, STEP, u_store=u_store)
        assert np.all(np.abs(Pg.cpu().numpy() - Pn) <= bP)
        assert np.all(np.abs(Qg.cpu().numpy() - Qn) <= bQ)
        assert abs(float(sse.item()) - s64) <= bs
    # ratings changed in place are the ones the next sweep reads
    d[2].fill_(3)
    d[5].fill_(3)
    C.cf_get_factors(h, Pg, Qg)
    P, Q = Pg.cpu().numpy().astype(np.float64), Qg.cpu().numpy().astype(np.float64)
    C.cf_sweep(h, 1, LAM, STEP, sse)
    three = np.full_like(rate, 3)
    s64 = O.cf_sweep_bound(U, I, off, item, three, ioff, iuser, three, P, Q, LAM, STEP,
                           u_store=u_store)
    assert abs(float(sse.item()) - s64[2]) <= s64[5]


def test_update_before_a_gather_only_decays(C, ratings):
    import torch
    U, I, off, item, rate = ratings
    d = _item_major(C, U, I, off, item, rate)
    rng = np.random.default_rng(1)
    P0, Q0 = (rng.random((n, 32)).astype(np.float32) for n in (U, I))
    Pg, Qg = torch.empty((U, 32), device="cuda"), torch.empty((I, 32), device="cuda")
    for sweeps in (3, 0):  # the second handle may get the memory that the first one used
        h = C.cf_create(U, I, 32, 0, *d)
        C.cf_set_factors(h, torch.as_tensor(P0).cuda(), torch.as_tensor(Q0).cuda())
        if sweeps:
            C.cf_sweep(h, sweeps, LAM, STEP)
            del h
    C.cf_sweep_phase(h, 2, LAM, STEP)
    C.cf_sweep_phase(h, 3, LAM, STEP)
    C.cf_get_factors(h, Pg, Qg)
    for got, x in ((Pg, P0), (Qg, Q0)):  # two products and a sum, rounded in FP32
        want = x.astype(np.float64) * (1.0 - STEP * LAM)
        assert np.all(np.abs(got.cpu().numpy() - want) <= 4 * 2.0 ** -24 * x)
