"""The bounded waits of the FP64 digit transform: a limit of one cycle makes the
first wait for a line's exponents or a stage run out.  The kernel then drains its
copies and MMAs, frees its tensor memory and returns, and the solve reports
FDI_ERR_TIMEOUT (no fault, the context stays usable); with the default limit
restored the same plan gives the bits of an untouched one."""
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


# 32 lines per item and fewer items than SMs; 64 lines and several items per CTA
@pytest.mark.parametrize("n", [(64, 64, 24), (160, 144, 64)])
def test_wait_limit_runs_out_then_fp64_plan_recovers(fdi, n):
    import torch
    faces = [tanh_faces(m, 1.5) for m in n]
    f = torch.from_numpy(np.ascontiguousarray(rhs_uniform(n[::-1], 5))).cuda()
    out, want = torch.empty_like(f), torch.empty_like(f)
    stream = torch.cuda.Stream()
    plan, fresh = fdi.plan_create(faces, n), fdi.plan_create(faces, n)
    torch.cuda.synchronize()
    try:
        fdi.helmholtz_solve(fresh, 1.0, f, want, stream)
        torch.cuda.synchronize()
        assert fdi.last_result(fresh)[3] == 0
        fdi.set_wait_limit(plan, 1)
        for _ in range(3):  # launch by launch, captured, replayed; the flag stays set
            fdi.helmholtz_solve(plan, 1.0, f, out, stream)
            torch.cuda.synchronize()
            with pytest.raises(fdi.FdiError) as e:
                fdi.last_result(plan)
            assert e.value.status == fdi.ERR_TIMEOUT
        fdi.set_wait_limit(plan, 0)
        for _ in range(3):
            out.zero_()
            torch.cuda.synchronize()
            fdi.helmholtz_solve(plan, 1.0, f, out, stream)
            torch.cuda.synchronize()
            assert fdi.last_result(plan)[3] == 0
            assert torch.equal(out, want)
    finally:
        plan.destroy()
        fresh.destroy()
