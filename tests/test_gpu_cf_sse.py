"""The squared-error sum of collaborative filtering outside the range of FP32: a
sum of FP64, so finite where single errors are; infinite, not NaN, where an error's
square is."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _one_rating_each(torch, C, U, K, precision, x):
    """U users that rated the one item with 5; every product p . q is x * x."""
    off = torch.arange(U + 1, dtype=torch.int64, device="cuda")
    item = torch.zeros(U, dtype=torch.int32, device="cuda")
    rate = torch.full((U,), 5, dtype=torch.uint8, device="cuda")
    ioff = torch.tensor([0, U], dtype=torch.int64, device="cuda")
    user = torch.arange(U, dtype=torch.int32, device="cuda")
    h = C.cf_create(U, 1, K, precision, off, item, rate, ioff, user, rate)
    P, Q = torch.zeros(U, K, device="cuda"), torch.zeros(1, K, device="cuda")
    P[:, 3] = x
    Q[:, 3] = x
    C.cf_set_factors(h, P, Q)
    sse = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    C.cf_sweep_phase(h, 0, 0.05, 1e-3, sse)
    return float(sse.item())


@pytest.mark.parametrize("K,precision", [(16, 0), (32, 0), (32, 1), (32, 2), (64, 0)])
def test_sum_beyond_fp32(K, precision):
    import torch
    from paper_1608_01362_gb300 import cagra as C
    U, x = 700_001, 2.0 ** 31
    want = U * (2.0 ** 62) ** 2  # 5 - 2^62 rounds to -2^62; every square 2^124, exact
    assert want > 3.5e38
    assert _one_rating_each(torch, C, U, K, precision, x) == want


@pytest.mark.parametrize("K,precision", [(16, 0), (32, 1), (32, 2), (64, 0)])
def test_square_beyond_fp32(K, precision):
    import torch
    from paper_1608_01362_gb300 import cagra as C
    assert _one_rating_each(torch, C, 1000, K, precision, 2.0 ** 40) == np.inf
