"""FP64 correction rounds.  A direct FP64 solve meets the default tolerance at its
first check, so a tolerance below rounding makes every round run: the transforms
that add to the solution, the residual's later checks, and, once the calls repeat,
the nested conditional bodies of the captured solve.  Launch by launch, captured
and replayed give the same bits."""
import numpy as np
import pytest

from oracle import assembled as asm
from workloads import rhs_uniform, tanh_faces

pytestmark = pytest.mark.gpu

ROUNDS = 3


@pytest.fixture(scope="module")
def fdi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_2461_gb300 import build
    build.build()
    import paper_1107_2461_gb300 as pkg
    return pkg


def run(fdi, plan, lam, rhs, out, stream):
    import torch
    out.zero_()
    torch.cuda.synchronize()
    if lam:
        fdi.helmholtz_solve(plan, lam, rhs, out, stream)
    else:
        fdi.laplace_solve(plan, rhs, out, stream)
    torch.cuda.synchronize()
    return fdi.last_result(plan)


# planes of up to 32 x 32 cells; digit products with 32 and with 64 lines per item; three
# eigen directions (small, digits, mixed); a permuted axis; the zero-flux Laplacian (small, digits)
@pytest.mark.parametrize("n,axis,wall,lam", [
    ((16, 20, 24), 2, 0, 0.5), ((40, 36, 33), 2, 0, 0.5), ((160, 144, 40), 2, 0, 1e-3), ((16, 20, 24), -1, 0, 0.5),
    ((40, 36, 33), -1, 0, 0.5), ((40, 36, 20), -1, 0, 0.5), ((40, 36, 33), 0, 0, 0.5), ((16, 20, 24), 2, 1, 0.0),
    ((40, 36, 33), 2, 1, 0.0), ((33, 20, 17), -1, 1, 0.0)])
def test_forced_rounds(fdi, n, axis, wall, lam):
    import torch
    faces = [tanh_faces(m, 1.5) for m in n]
    plan = fdi.plan_create(faces, n, (wall,) * 3, (wall,) * 3, thomas_axis=axis)
    eager = fdi.plan_create(faces, n, (wall,) * 3, (wall,) * 3, thomas_axis=axis)
    fdi.set_graphs(eager, False)
    stream = torch.cuda.Stream()
    rhs = torch.from_numpy(np.ascontiguousarray(rhs_uniform(n[::-1], 3))).cuda()
    out, want = torch.empty_like(rhs), torch.empty_like(rhs)
    try:
        _, steps, rel0, status = run(fdi, eager, lam, rhs, want, stream)
        assert status == 0 and steps == 0
        for p in (plan, eager):
            p.set_tolerances(1e-30, ROUNDS, 1e-11, 100)
        for seed in (3, 3, 4, 5):  # launch by launch, captured, replayed with other values
            rhs.copy_(torch.from_numpy(np.ascontiguousarray(rhs_uniform(n[::-1], seed))))
            _, steps, rel, status = run(fdi, eager, lam, rhs, want, stream)
            assert status == fdi.ERR_NOT_CONVERGED and steps == ROUNDS
            # a correction of the wrong sign would double the residual in every round
            assert rel <= 2 * rel0
            _, steps, rel_g, status = run(fdi, plan, lam, rhs, out, stream)
            assert status == fdi.ERR_NOT_CONVERGED and steps == ROUNDS and rel_g == rel
            assert torch.equal(out, want), seed
        # and with the tolerance back no round runs
        plan.set_tolerances(1e-11, ROUNDS, 1e-11, 100)
        for _ in range(3):
            _, steps, _, status = run(fdi, plan, lam, rhs, out, stream)
            assert status == 0 and steps == 0
    finally:
        plan.destroy()
        eager.destroy()
    if lam and n[0] < 100:
        ops = asm.cell_ops(faces, (0, 0, 0), (0, 0, 0))
        f, got = rhs.cpu().numpy(), want.cpu().numpy()
        assert asm.relative_residual(ops, got, f, lam) <= 1e-11


def test_forced_rounds_on_a_cylinder_and_in_batches(fdi):
    import torch
    stream = torch.cuda.Stream()
    sizes = [(40, 36, 33), (16, 20, 24), (65, 30, 17)]
    make = [lambda n=n: fdi.plan_create([tanh_faces(m, 1.5) for m in n], n) for n in sizes]
    make.append(lambda: fdi.plan_create_cyl(0.5 + tanh_faces(33, 1.0), 40, tanh_faces(36, 1.0)))
    plans, eager = [f() for f in make], [f() for f in make]
    for p in plans + eager:
        p.set_tolerances(1e-30, ROUNDS, 1e-11, 100)
    for p in eager:
        fdi.set_graphs(p, False)
    # the first plan twice in the batch: its rounds follow one another on a stream
    order, lams = [0, 1, 2, 3, 0], [0.5, 0.01, 1.0, 0.3, 0.02]
    shapes = [(33, 36, 40), (24, 20, 16), (17, 30, 65), (36, 40, 33)]
    rhs = [torch.zeros(shapes[q], dtype=torch.float64, device="cuda") for q in order]
    outs, want = [torch.empty_like(r) for r in rhs], [torch.empty_like(r) for r in rhs]
    try:
        for seed in (1, 1, 2, 3):
            for k, r in enumerate(rhs):
                r.copy_(torch.from_numpy(np.ascontiguousarray(rhs_uniform(tuple(r.shape), 10 * seed + k))))
                _, steps, _, _ = run(fdi, eager[order[k]], lams[k], r, want[k], stream)
                assert steps == ROUNDS
                outs[k].zero_()
            torch.cuda.synchronize()
            fdi.helmholtz_solve_batched([plans[q] for q in order], lams, rhs, outs, stream)
            torch.cuda.synchronize()
            for k in range(len(order)):
                assert fdi.last_result(plans[order[k]])[1] == ROUNDS
                assert torch.equal(outs[k], want[k]), (seed, k)
    finally:
        for p in plans + eager:
            p.destroy()
