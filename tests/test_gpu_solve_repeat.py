"""The step that converges raises the stop flag while the same launch's other
blocks start: a solve's bits and counts must not depend on when they read it."""
import pytest

from gpu_util import Plan
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [0.0, 2.0])
@pytest.mark.parametrize("restart", [1, 4, 30])
def test_solves_repeat(restart, k):
    import torch
    m = I.icosphere(5 if not k else 4)               # 41 (81 complex) blocks and more in the last kernel of a step
    P = Plan(m, bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE, k, p=6, leaf_size=32, precision=bem.BEM_MIXED)
    dt = torch.complex128 if k else torch.float64
    chi = torch.tensor(I.random_vector(P.n_chi, 90, bool(k)), device="cuda", dtype=dt)
    sp = bem.bem_solve_params_default(restart=restart, tol=1e-6, max_iter=60)
    batch = bem.bem_batch_create(P.ctx, 1)
    group = bem.bem_group_create(P.ctx, [P.plan])
    seen = []
    for i in range(12):
        phi = torch.full((P.n_phi,), float("nan"), device="cuda", dtype=dt)
        _, (info,) = bem.bem_solve(P.plan, chi, phi, 1, sp)
        torch.cuda.synchronize()
        seen.append((phi, info.iters, info.restarts))
    for i in range(4):
        phi = torch.full((P.n_phi,), float("nan"), device="cuda", dtype=dt)
        torch.cuda.synchronize()
        slot = bem.bem_batch_submit(batch, P.plan, chi, phi, sp)
        bem.bem_batch_wait(batch, slot)
        info = bem.bem_batch_poll(batch, slot)[1]
        bem.bem_batch_release(batch, slot)
        seen.append((phi, info.iters, info.restarts))
        phi = torch.full((P.n_phi,), float("nan"), device="cuda", dtype=dt)
        torch.cuda.synchronize()
        _, (info,), _ = bem.bem_group_solve(group, [chi], [phi], sp)
        seen.append((phi, info.iters, info.restarts))
    assert torch.isfinite(torch.view_as_real(seen[0][0]) if k else seen[0][0]).all()
    for phi, iters, restarts in seen[1:]:
        assert (iters, restarts) == seen[0][1:]
        assert torch.equal(phi, seen[0][0])
    bem.bem_group_destroy(group)
    bem.bem_batch_destroy(batch)
    P.close()
