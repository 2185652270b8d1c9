"""Solves that a caller captures into a graph of their own after the same calls ran
on that stream: the library then keeps graphs for these arguments, and none of
them may enter the caller's capture (nor may the library begin a capture inside
it).  Every replay gives the bits of a plan without graphs, and the kept graphs
still replay afterwards."""
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


def fill(t, seed):
    import torch
    t.copy_(torch.from_numpy(np.ascontiguousarray(rhs_uniform(tuple(t.shape), seed))))
    torch.cuda.synchronize()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("warm", [0, 1, 2, 3])  # nothing kept; arguments seen; graph kept; graph replayed
def test_field_solve_captured_by_the_caller(fdi, prec, warm):
    import torch
    n = (40, 36, 33)
    p = fdi.PREC_FP64 if prec == "fp64" else fdi.PREC_MIXED_F16
    plan = fdi.plan_create(box_faces(n, 1.5), n, prec=p)
    ref_plan = fdi.plan_create(box_faces(n, 1.5), n, prec=p)
    fdi.set_graphs(ref_plan, False)
    rhs = torch.zeros(n[::-1], dtype=torch.float64, device="cuda")
    out, ref = torch.empty_like(rhs), torch.empty_like(rhs)
    fill(rhs, 1)
    stream = torch.cuda.Stream()
    for _ in range(warm):
        fdi.helmholtz_solve(plan, 0.5, rhs, out, stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        fdi.helmholtz_solve(plan, 0.5, rhs, out, stream)
        fdi.helmholtz_solve(plan, 0.5, rhs, out, stream)  # the same arguments again inside one capture
    for seed in range(2, 5):
        fill(rhs, seed)
        fdi.helmholtz_solve(ref_plan, 0.5, rhs, ref)
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert fdi.last_result(plan)[3] == 0
        assert torch.equal(out, ref), seed
        for _ in range(2):
            out.zero_()
            torch.cuda.synchronize()
            fdi.helmholtz_solve(plan, 0.5, rhs, out, stream)
            torch.cuda.synchronize()
            assert torch.equal(out, ref), seed
    del graph
    plan.destroy()
    ref_plan.destroy()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("warm", [0, 1, 3])
def test_batch_captured_by_the_caller(fdi, prec, warm):
    import torch
    p = fdi.PREC_FP64 if prec == "fp64" else fdi.PREC_MIXED_F16
    sizes = [(40, 36, 33), (16, 20, 24), (65, 30, 17)]
    lams = [0.5, 0.01, 1.0]
    plans = [fdi.plan_create(box_faces(n, 1.5), n, prec=p) for n in sizes]
    rhs = [torch.zeros(n[::-1], dtype=torch.float64, device="cuda") for n in sizes]
    outs, refs = [torch.empty_like(r) for r in rhs], [torch.empty_like(r) for r in rhs]
    ref_plans = [fdi.plan_create(box_faces(n, 1.5), n, prec=p) for n in sizes]
    for q in ref_plans:
        fdi.set_graphs(q, False)
    for q, r in enumerate(rhs):
        fill(r, q)
    stream = torch.cuda.Stream()
    for _ in range(warm):
        fdi.helmholtz_solve_batched(plans, lams, rhs, outs, stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        fdi.helmholtz_solve_batched(plans, lams, rhs, outs, stream)
    for seed in (10, 20):
        for q, r in enumerate(rhs):
            fill(r, seed + q)
            fdi.helmholtz_solve(ref_plans[q], lams[q], r, refs[q])
            outs[q].zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for q in range(len(sizes)):
            assert fdi.last_result(plans[q])[3] == 0
            assert torch.equal(outs[q], refs[q]), (seed, q)
            outs[q].zero_()
        torch.cuda.synchronize()
        fdi.helmholtz_solve_batched(plans, lams, rhs, outs, stream)
        torch.cuda.synchronize()
        for q in range(len(sizes)):
            assert torch.equal(outs[q], refs[q]), (seed, q)
    del graph
    for q in plans + ref_plans:
        q.destroy()
