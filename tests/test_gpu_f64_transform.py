"""FP64 eigenvector transforms (digit products on the tensor cores, plain FP64 on
small planes) at the edges of their tiles: 16-column steps, 128-mode tiles, 32 and
64 lines per item, planes of up to 32 x 32 cells.

With lambda = 0 the operator is the identity, so a solve is the forward and
back transforms alone: u must equal f.  z-planes do not mix then, and each one
is given its own scale, a single entry or nothing, so a result is judged
against its own plane.  Tolerance: 64 n 2^-53 of the plane's largest value (n
the longer transformed direction): E E^{-1} = I holds to a few n 2^-53 with the
eigenbasis computed in FP64, the basis' condition is at most 4 at this
stretching, and the transforms add less than an FP64 dot product."""
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


def solve(fdi, plan, lam, f):
    import torch
    rhs = torch.from_numpy(np.ascontiguousarray(f)).cuda()
    out = torch.empty_like(rhs)
    fdi.helmholtz_solve(plan, lam, rhs, out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("n", [(2, 3, 5), (15, 16, 6), (17, 33, 5), (31, 64, 5), (65, 63, 9), (127, 129, 5),
                               (128, 130, 60), (40, 200, 61), (255, 256, 5), (256, 241, 5),
                               # both plane transforms (and the z steps) in one launch up to 32 cells
                               (32, 32, 32), (32, 31, 33), (33, 32, 32), (3, 30, 17)])
@pytest.mark.parametrize("axis", [2, -1])
def test_transforms_invert_each_other(fdi, n, axis):
    faces = [tanh_faces(n[d], 1.5) for d in range(3)]
    plan = fdi.plan_create(faces, n, thomas_axis=axis)
    f = rhs_uniform(n[::-1], 5)
    if axis == 2:
        rng = np.random.default_rng(6)
        f *= (10.0 ** rng.integers(-12, 13, size=n[2]))[:, None, None]
        f[1] = 0.0
        f[2] = 0.0
        f[2, n[1] // 2, n[0] - 1] = -3.0e7
    try:
        got = solve(fdi, plan, 0.0, f)
    finally:
        plan.destroy()
    tol = 64 * max(n[:2] if axis == 2 else n) * 2.0**-53
    planes = range(n[2]) if axis == 2 else [slice(None)]
    for k in planes:
        assert np.abs(got[k] - f[k]).max() <= tol * np.abs(f[k]).max(), k


@pytest.mark.parametrize("k", [300, -300])
def test_power_of_two_scaling_is_exact(fdi, k):
    # every line carries its own exponent: scaling the right-hand side by a
    # power of two scales the solution by it, to the last bit
    n = (45, 70, 13)
    plan = fdi.plan_create([tanh_faces(n[d], 1.5) for d in range(3)], n)
    f = rhs_uniform(n[::-1], 7)
    try:
        a = solve(fdi, plan, 0.3, f)
        b = solve(fdi, plan, 0.3, np.ldexp(f, k))
    finally:
        plan.destroy()
    assert np.array_equal(np.ldexp(a, k), b)


@pytest.mark.parametrize("n", [(31, 7, 2), (32, 8, 8), (33, 9, 9), (64, 8, 17), (65, 16, 3), (97, 17, 5), (2, 2, 33)])
@pytest.mark.parametrize("walls", [(0, 0), (1, 1), (0, 1), (1, 0)])
def test_residual_confirms_the_first_solve(fdi, n, walls):
    # columns, rows and planes at the edges of the residual's blocks: a face or
    # a wall missed there would leave a residual of order one, so the first check
    # of a direct solve confirms it at the FP64 tolerance with no correction
    import torch
    plan = fdi.plan_create([tanh_faces(n[d], 1.5) for d in range(3)], n, (walls[0],) * 3, (walls[1],) * 3)
    try:
        for lam in (0.7, 0.0) if walls != (1, 1) else (0.7,):
            f = torch.from_numpy(rhs_uniform(n[::-1], 3)).cuda()
            out = torch.empty_like(f)
            if lam:
                fdi.helmholtz_solve(plan, lam, f, out)
            else:
                fdi.laplace_solve(plan, f, out)
            torch.cuda.synchronize()
            _, steps, rel, status = fdi.last_result(plan)
            assert status == 0 and steps == 0 and rel <= 1e-11
    finally:
        plan.destroy()


@pytest.mark.parametrize("n", [(31, 3, 33), (64, 9, 8), (5, 33, 70)])  # r, theta, z
def test_residual_confirms_the_first_cylindrical_solve(fdi, n):
    import torch
    plan = fdi.plan_create_cyl(0.5 + tanh_faces(n[0], 1.0), n[1], tanh_faces(n[2], 1.0))
    f = torch.from_numpy(rhs_uniform(n[::-1], 3)).cuda()
    out = torch.empty_like(f)
    try:
        fdi.helmholtz_solve(plan, 0.3, f, out)
        torch.cuda.synchronize()
        _, steps, rel, status = fdi.last_result(plan)
    finally:
        plan.destroy()
    assert status == 0 and steps == 0 and rel <= 1e-11
