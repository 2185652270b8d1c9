"""FP32 line sweep on the singular zero-flux Laplacian: the pair of lines with the
null line, solved by a block of its own in the two-lines-per-thread configurations
(2, 3), against the one-line-per-thread sweep (64), which keeps it among the
others.  The arithmetic is the same operation by operation, so the solutions are
the same bits.  Sizes: the smallest plan, odd numbers of lines along y, partial
and whole blocks of 16 planes, one and several blocks of pairs, the longest line."""
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


@pytest.mark.parametrize("n", [(2, 2, 2), (3, 2, 16), (5, 7, 17), (16, 8, 15), (33, 13, 48), (64, 64, 64),
                               (20, 31, 128), (9, 12, 255), (12, 10, 256)])
def test_null_line_block_matches_single_line_sweep(fdi, n):
    import torch
    neumann = (fdi.BC_NEUMANN,) * 3
    plan = fdi.plan_create([tanh_faces(m, 1.5) for m in n], n, prec=fdi.PREC_MIXED_F16, bc_lo=neumann,
                           bc_hi=neumann)
    fdi.set_resident(plan, False)
    f = torch.from_numpy(np.ascontiguousarray(rhs_uniform(n[::-1], 11))).cuda()
    outs = []
    for config in (64, 2, 3):
        fdi.set_thomas_config(plan, config)
        out = torch.empty_like(f)
        fdi.laplace_solve(plan, f, out)
        torch.cuda.synchronize()
        outs.append(out)
    plan.destroy()
    assert torch.isfinite(outs[0]).all() and outs[0].abs().max() > 0
    assert torch.equal(outs[1], outs[0]) and torch.equal(outs[2], outs[0])
