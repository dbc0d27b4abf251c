"""A call whose host side waits for a kernel's result leaves the core alone when
other work is long in front of it on the stream, and later calls find no error
left behind."""
import time

import pytest

import graphgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["lp_run", "bc_run"])
def test_host_sleeps_behind_a_long_queue(call):
    import torch
    from paper_1608_01362_gb300 import cagra as C, pipeline as P
    g = graphgen.rmat(9, 8, seed=4, symmetric=True)
    graph = P.Graph(g.offsets, g.src, cluster_mode=None)
    if call == "lp_run":
        seg = C.pr_build_segments(graph.offsets, graph.src, 2)
        lab = torch.arange(g.V, dtype=torch.int32, device="cuda")
        run = lambda: C.lp_run(seg, lab)  # noqa: E731
    else:
        b = P.Betweenness(graph)
        run = lambda: C.bc_run(b.h, [0], b.bc)  # noqa: E731
    run()
    torch.cuda.synchronize()
    torch.cuda._sleep(1_600_000_000)  # 0.8 s at 2 GHz; the kernel ends by itself
    wall, cpu = time.perf_counter(), time.thread_time()
    run()
    wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
    assert wall > 0.3 and cpu < 0.4 * wall, (wall, cpu)
    C.cg_inv_outdeg(graph.outdeg, graph.inv)
    torch.cuda.synchronize()
