"""The admission estimate bounds a plan's peak where its per-node part dominates:
many small leaves, an uneven body, 3-node triangles, and the largest measured mesh."""
import pytest

from gpu_util import Plan
from paper_0908_0673_gb300 import bem, inputs as I
from paper_0908_0673_gb300.serve import estimate_peak_footprint

pytestmark = pytest.mark.gpu

MESHES = {
    "cube15": lambda: I.cube(15), "ell30": lambda: I.geodesic(30, axes=(0.5, 1.0, 2.0)), "geo64": lambda: I.geodesic(64),
    "ell80-tri3": lambda: I.geodesic(80, I.TRI3, axes=(0.5, 1.0, 2.0)),
}


@pytest.mark.parametrize("precision", [bem.BEM_F64, bem.BEM_MIXED], ids=["f64", "mixed"])
@pytest.mark.parametrize("k", [0.0, 4.0])
@pytest.mark.parametrize("mesh,leaf", [("cube15", 32), ("ell30", 32), ("geo64", 64), ("ell80-tri3", 64)])
def test_estimate_bounds_peak(mesh, leaf, k, precision):
    import torch
    m = MESHES[mesh]()
    green = bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE
    P = Plan(m, green, k, p=10, leaf_size=leaf, eta=2.0, precision=precision)
    dt = torch.complex128 if k else torch.float64
    chi, phi = torch.ones(P.n_chi, device="cuda", dtype=dt), torch.empty(P.n_phi, device="cuda", dtype=dt)
    bem.bem_solve(P.plan, chi, phi, 1, bem.bem_solve_params_default(max_iter=2))
    peak, est = bem.bem_plan_peak_footprint(P.plan), estimate_peak_footprint(m.n_nodes, green, precision)
    P.close()
    assert peak <= est, (peak / 1e6, est / 1e6)
