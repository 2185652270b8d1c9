"""FP64 solves at the ends of FP64's exponent range, which scaled problems reach:
what the plain formulas represent, the kernels have to keep."""
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


@pytest.mark.parametrize("n", [(40, 36, 33), (16, 20, 24)])  # digit products, small planes
def test_line_pivots_below_the_normal_range(fdi, n):
    # -lambda Delta u = f with lambda = 2^-1028: the pivots of the line sweep run
    # from 2^-1023.7 to 2^-1015 here, on both sides of the smallest normal number
    # 2^-1022, and their reciprocals are finite (a pivot below 2^-1024 has none).
    # The solution is 2^1028 times that for lambda = 1.  Tolerance: the sweep's
    # coefficients, at least 2^-1024, carry a relative error of 2^-51 instead of
    # 2^-53, amplified by at most the operator's condition number, 4.4e3.
    import torch
    plan = fdi.plan_create([tanh_faces(m, 1.5) for m in n], n)
    f = torch.from_numpy(np.ascontiguousarray(rhs_uniform(n[::-1], 3))).cuda()
    small = f * 2.0**-200
    want, got = torch.empty_like(f), torch.empty_like(f)
    try:
        fdi.field_solve(plan, fdi.FIELD_CELL, 0.0, 1.0, f, want)
        torch.cuda.synchronize()
        assert fdi.last_result(plan)[3] == 0
        fdi.field_solve(plan, fdi.FIELD_CELL, 0.0, 2.0**-1028, small, got)
        torch.cuda.synchronize()
        _, _, rel, status = fdi.last_result(plan)
    finally:
        plan.destroy()
    assert status == 0 and rel <= 1e-11
    got = np.ldexp(got.cpu().numpy(), 200 - 1028)
    want = want.cpu().numpy()
    assert np.abs(got - want).max() <= 2.0**-51 * 4.4e3 * np.abs(want).max()


@pytest.mark.parametrize("n", [(40, 36, 33), (130, 17, 9), (16, 20, 24)])  # digit products (two), small planes
@pytest.mark.parametrize("k", [-1015, -1030])  # lines with some subnormal entries; with nothing else
def test_subnormal_entries_count(fdi, n, k):
    # lambda = 0: the solve is the forward and back transforms with a division by
    # M_z between products with it, u = f.  Tolerance: the relative part of the
    # other transform tests, and half of the subnormal spacing 2^-1074 for every
    # step that rounds there, carried through the later steps by the matrices' row sums.
    import torch
    plan = fdi.plan_create([tanh_faces(m, 1.5) for m in n], n)
    f = np.ldexp(rhs_uniform(n[::-1], 7), k)
    rhs = torch.from_numpy(np.ascontiguousarray(f)).cuda()
    out = torch.empty_like(rhs)
    try:
        (_, ex, _), (_, ey, eyi) = [plan.eigen(fdi.FIELD_CELL, d) for d in (0, 1)]
        fdi.helmholtz_solve(plan, 0.0, rhs, out)
        torch.cuda.synchronize()
        assert fdi.last_result(plan)[3] == 0
    finally:
        plan.destroy()
    half = 2.0**-1055  # half a spacing; in units of 2^-20 from here
    norm = [np.abs(e).sum(axis=1).max() for e in (ex, ey, eyi)]
    err = (half * norm[2] + 2 * half) / np.diff(tanh_faces(n[2], 1.5)).min() + half
    err = (err * norm[1] + half) * norm[0] + half
    tol = 64 * max(n[:2]) * 2.0**-53 * np.abs(f).max() * 2.0**20 + err
    assert np.abs(np.ldexp(out.cpu().numpy() - f, 20)).max() <= tol
