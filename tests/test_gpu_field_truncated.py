"""Far fields against the truncated multipole sum itself, coefficient for coefficient.

One box, points beyond eta times its radius: the field is the degree-p
polynomial a(d) G(x - c) of the oracle's moments and derivatives, whatever
basis evaluates it, so a wrong or missing coefficient shows at any order.
Tolerances: float64 1e-11 (sums of some 1e3 terms in 48 bits and more), mixed
2e-6 (float32 moments)."""
from math import factorial

import numpy as np
import pytest

from gpu_util import Plan, rel_l2
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [0.0, 1.5])
@pytest.mark.parametrize("p", [1, 2, 3, 6, 11, 20])
@pytest.mark.parametrize("precision,tol", [(bem.BEM_F64, 1e-11), (bem.BEM_MIXED, 2e-6)])
def test_equals_truncated_sum(oracle_lib, precision, tol, p, k):
    O = oracle_lib
    m = I.icosphere(1, I.TRI6)
    green = bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE
    P = Plan(m, green, k, p=p, leaf_size=4000, eta=2.0, precision=precision)
    T = bem.bem_plan_export_tree(P.plan)
    c = T["centre"][0]
    rng = np.random.default_rng(11)
    phi, chi = I.random_vector(P.n_phi, 12, bool(k)), I.random_vector(P.n_chi, 13, bool(k))
    d = rng.standard_normal((37, 3))
    pts = c + d / np.linalg.norm(d, axis=1, keepdims=True) * np.geomspace(2.2, 30.0, 37)[:, None] * T["radius"][0]
    qx, qn, qw, qL = O.quad_points(m.nodes, m.elems)
    e = np.repeat(np.arange(m.n_elems), 7)
    M = O.p2m(p, c, qx, qn, -qw * (qL * chi[P.chi_idx[e]]).sum(1), qw * (qL * phi[m.elems[e]]).sum(1))
    w = np.array([(-1.0) ** a.sum() / np.prod([float(factorial(i)) for i in a]) for a in O.mindex(p)])
    ref = np.array([(w * M * O.green_derivs(p, x - c, green, k)).sum() for x in pts])
    u = P.torch.empty(len(pts), device="cuda", dtype=P.torch.complex128 if k else P.torch.float64)
    bem.bem_field(P.plan, P._dev(phi), P._dev(chi), P.torch.tensor(pts, device="cuda"), u)
    got = u.cpu().numpy()
    assert np.all(np.abs(got - (ref if k else ref.real)) < tol * np.abs(ref).max() * (2.2 * T["radius"][0] / np.linalg.norm(pts - c, axis=1)) ** 0.5)
    P.close()


@pytest.mark.parametrize("k", [0.0, 2.0])
def test_small_strengths_beside_large_ones(k):
    """Large values on a flat face leave nothing at the face's other nodes (r . n = 0 to 2^-53), where
    values 1e-8 as large elsewhere must keep their digits: 1e-16 / 1e-8 times some hundred terms, 1e-6."""
    m = I.cube(2, I.TRI6, grade=0.0)
    P = Plan(m, bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE, k, p=8, leaf_size=128)
    inner = np.where((m.nodes[:, 2] == m.nodes[:, 2].max()) & (np.abs(m.nodes[:, :2]).max(1) < 0.99))[0]
    assert len(inner) >= 8
    small = I.random_vector(P.n_phi, 14, bool(k)) * 1e-8
    both = small.copy()
    small[inner[::2]] = 0.0
    both[inner[::2]] = 1.0
    at = inner[1::2]
    assert rel_l2(P.matvec(bem.BEM_OP_A, both)[at], P.matvec(bem.BEM_OP_A, small)[at]) < 1e-6
    P.close()
