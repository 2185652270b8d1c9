"""Repeated calls that the library replays as graphs, among other work of the
caller: solves on the default stream between default-stream operations that change
their input and read their output, and batches that alternate, more of them than
are kept, also after a plan of a kept one is gone.  Reference: plans without graphs."""
import numpy as np
import pytest

from workloads import rhs_uniform, tanh_faces

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


def plan_of(fdi, n, prec, graphs=True):
    plan = fdi.plan_create([tanh_faces(m, 1.5) for m in n], n,
                           prec=fdi.PREC_FP64 if prec == "fp64" else fdi.PREC_MIXED_F16)
    fdi.set_graphs(plan, graphs)
    return plan


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("batch", [False, True])
def test_default_stream_replays_in_order_with_other_work(fdi, prec, batch):
    import torch
    n = (65, 36, 33)
    plan, eager = plan_of(fdi, n, prec), plan_of(fdi, n, prec, False)
    base = torch.from_numpy(np.ascontiguousarray(rhs_uniform(n[::-1], 1))).cuda()
    rhs, out = torch.empty_like(base), torch.empty_like(base)
    ref_in, ref = torch.empty_like(base), torch.empty_like(base)
    kept, wants = [], []
    scratch = torch.randn(1 << 24, device="cuda")  # work ahead of each solve
    for k in range(6):  # no synchronisation in between
        scratch.mul_(1.0001)
        torch.mul(base, float(k + 1), out=rhs)
        if batch:
            fdi.helmholtz_solve_batched([plan], [0.5], [rhs], [out])
        else:
            fdi.helmholtz_solve(plan, 0.5, rhs, out)
        kept.append(out.clone())
        rhs.zero_()
        out.zero_()
    for k in range(6):
        torch.mul(base, float(k + 1), out=ref_in)
        fdi.helmholtz_solve(eager, 0.5, ref_in, ref)
        wants.append(ref.clone())
    torch.cuda.synchronize()
    for k in range(6):
        assert torch.equal(kept[k], wants[k]), k
    plan.destroy()
    eager.destroy()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_alternating_batches(fdi, prec):
    import torch
    sizes = [(40, 36, 33), (16, 20, 24), (33, 30, 17)]
    lams = [0.5, 0.01, 1.0]
    plans = [plan_of(fdi, n, prec) for n in sizes]
    eager = [plan_of(fdi, n, prec, False) for n in sizes]
    stream = torch.cuda.Stream()
    sets = []
    for b in range(5):
        rhs = [torch.zeros(n[::-1], dtype=torch.float64, device="cuda") for n in sizes]
        sets.append((rhs, [torch.empty_like(r) for r in rhs]))
    ref = [torch.empty_like(r) for r in sets[0][0]]
    seed = 0

    def check(b):
        nonlocal seed
        rhs, outs = sets[b]
        for q, r in enumerate(rhs):
            seed += 1
            r.copy_(torch.from_numpy(np.ascontiguousarray(rhs_uniform(tuple(r.shape), seed))))
            outs[q].zero_()
        torch.cuda.synchronize()
        fdi.helmholtz_solve_batched(plans, lams, rhs, outs, stream)
        torch.cuda.synchronize()
        for q in range(len(sizes)):
            assert fdi.last_result(plans[q])[3] == 0
            fdi.helmholtz_solve(eager[q], lams[q], rhs[q], ref[q], stream)
            torch.cuda.synchronize()
            assert torch.equal(outs[q], ref[q]), (b, q)

    for b in (0, 1) * 4:
        check(b)
    for b in (0, 1, 2, 3, 4) * 3 + (4, 4, 0, 0, 0):
        check(b)
    # a plan of the kept batches goes, another takes its place (often its address)
    plans[1].destroy()
    plans[1] = plan_of(fdi, sizes[1], prec)
    for b in (4, 0, 4, 0, 4, 0):
        check(b)
    # a changed control drops the kept batches of its plan only
    plans[0].set_tolerances(1e-10, 2, 1e-10, 100)
    eager[0].set_tolerances(1e-10, 2, 1e-10, 100)
    for b in (4, 0, 4, 0):
        check(b)
    for p in plans + eager:
        p.destroy()
