"""Segment plans with room for few segments: always a partition of [0, V) in 1 to
k_max segments."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k_max", [1, 2, 3, 4])
@pytest.mark.parametrize("V", [1, 2, 33, 5000])
@pytest.mark.parametrize("smem", [0, 16, 600])
def test_plan_is_a_partition(V, smem, k_max):
    import torch
    from paper_1608_01362_gb300 import cagra as C
    rng = np.random.default_rng(V)
    deg = np.sort(rng.integers(0, 40, V))[::-1].astype(np.int32).copy()
    for tail in (0, 1, V // 3, V):
        deg[V - tail:] = 0
        b = C.pr_plan_bounds(torch.as_tensor(deg).cuda(), smem, 10.0, 100, k_max)
        assert 1 <= len(b) - 1 <= k_max, b
        assert b[0] == 0 and b[-1] == V and np.all(np.diff(b) >= 0), b


@pytest.mark.parametrize("smem", [0, 100, 512, 5000])
def test_sums_from_a_copy_and_from_the_device(smem):
    """65,536 vertices are summed on the host, one more on the device: a vertex
    without edges behind them only adds a last segment."""
    import torch
    from paper_1608_01362_gb300 import cagra as C
    deg = np.sort(np.random.default_rng(3).integers(1, 40, 65536))[::-1].astype(np.int32).copy()
    few = C.pr_plan_bounds(torch.as_tensor(deg).cuda(), smem, 10.0, 5000)
    more = C.pr_plan_bounds(torch.as_tensor(np.append(deg, 0).astype(np.int32)).cuda(), smem, 10.0,
                            5000)
    assert len(few) > 3 and more.tolist() == few.tolist() + [65537]
