"""Products whose output overlaps their input: the same bits as into memory of their own."""
import numpy as np
import pytest

from gpu_util import Plan
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu


def _stages(plan, op, x, y):
    bem.bem_plan_stage_times(plan, op, x, y, 1)


@pytest.mark.parametrize("form", [bem.bem_matvec, bem.bem_matvec_noalloc, _stages], ids=["graph", "noalloc", "stages"])
@pytest.mark.parametrize("k", [0.0, 2.0])
@pytest.mark.parametrize("precision", [bem.BEM_F64, bem.BEM_MIXED], ids=["f64", "mixed"])
def test_output_over_input(precision, k, form):
    import torch
    P = Plan(I.cube(6, I.TRI6), bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE, k, p=8, leaf_size=32, eta=2.0,
             precision=precision)
    dt = torch.complex128 if k else torch.float64
    for op, n in ((bem.BEM_OP_A, P.n_phi), (bem.BEM_OP_B, P.n_chi)):
        x = torch.tensor(I.random_vector(n, 70 + op, bool(k)), device="cuda", dtype=dt)
        ref = torch.empty(P.n_phi, device="cuda", dtype=dt)
        form(P.plan, op, x, ref)
        for off in (0, 5):                       # the same memory, and shifted by some entries
            for _ in range(10):
                buf = torch.empty(max(n, P.n_phi) + off, device="cuda", dtype=dt)
                buf[:n] = x
                y = buf[off:off + P.n_phi]
                form(P.plan, op, buf[:n], y)
                torch.cuda.synchronize()
                assert torch.equal(y, ref), (op, off)
    P.close()
