"""Solves called by one thread while another captures a graph of its own (global
mode, PyTorch's default): the graphs that the library builds for repeated calls must
not invalidate that capture, and the solves give their usual bits."""
import threading

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


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("call", ["default", "own", "batch_default", "batch_own"])
def test_repeated_solves_beside_another_threads_capture(fdi, prec, call):
    import torch
    n = (40, 36, 33)
    p = fdi.PREC_FP64 if prec == "fp64" else fdi.PREC_MIXED_F16
    plan = fdi.plan_create(box_faces(n, 1.5), n, prec=p)
    ref_plan = fdi.plan_create(box_faces(n, 1.5), n, prec=p)
    fdi.set_graphs(ref_plan, False)
    rhs = torch.from_numpy(np.ascontiguousarray(rhs_uniform(n[::-1], 1))).cuda()
    out, ref = torch.empty_like(rhs), torch.empty_like(rhs)
    own = torch.cuda.Stream()
    stream = 0 if call.endswith("default") else own
    # kernels are loaded and the batch's streams made before the capture begins
    fdi.helmholtz_solve(ref_plan, 0.5, rhs, ref, stream)
    fdi.helmholtz_solve_batched([ref_plan], [0.5], [rhs], [ref], stream)
    x = torch.arange(1000.0, device="cuda")
    torch.cuda.synchronize()
    errors, go, done = [], threading.Event(), threading.Event()

    def solves():
        go.wait(60)
        try:
            for _ in range(4):  # launch by launch, captured, replayed
                if call.startswith("batch"):
                    fdi.helmholtz_solve_batched([plan], [0.5], [rhs], [out], stream)
                else:
                    fdi.helmholtz_solve(plan, 0.5, rhs, out, stream)
        except Exception as e:
            errors.append(e)
        done.set()

    t = threading.Thread(target=solves)
    t.start()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        y = x + 1
        go.set()
        assert done.wait(60)
        y = y * 2
    t.join()
    assert not errors
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, (x + 1) * 2)
    assert torch.equal(out, ref)
    del graph
    plan.destroy()
    ref_plan.destroy()
