"""An FP64 solve enqueued into a graph that the caller captures: plain launches
(the library's conditional refinement rounds belong to its own graphs only), the
same bits on every replay as the eager solve."""
import numpy as np
import pytest

from workloads import box_faces, rhs_uniform

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fdi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_2461_gb300 import build
    build.build()
    import paper_1107_2461_gb300 as pkg
    return pkg


@pytest.mark.parametrize("n", [(20, 24, 16), (40, 36, 33)])
def test_fp64_solve_in_a_callers_capture(fdi, n):
    import torch
    plan = fdi.plan_create(box_faces(n, 1.5), n, prec=fdi.PREC_FP64)
    ref_plan = fdi.plan_create(box_faces(n, 1.5), n, prec=fdi.PREC_FP64)
    fdi.set_graphs(ref_plan, False)
    rhs = torch.zeros(n[::-1], dtype=torch.float64, device="cuda")
    out, ref = torch.empty_like(rhs), torch.empty_like(rhs)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fdi.helmholtz_solve(plan, 0.5, rhs, out)
    for seed in range(3):
        rhs.copy_(torch.from_numpy(np.ascontiguousarray(rhs_uniform(n[::-1], seed))))
        graph.replay()
        fdi.helmholtz_solve(ref_plan, 0.5, rhs, ref)
        torch.cuda.synchronize()
        assert fdi.last_result(plan)[3] == 0
        assert torch.equal(out, ref), seed
    del graph
    plan.destroy()
    ref_plan.destroy()
