"""Edges of the field evaluation: orders 1 to 20, the subdivision depth from
none to its limit, point counts off the block size, a tree of tiny leaves with
level-dependent orders, and points from almost on the surface to far away.

Tolerances: a mesh in one box near its points has no far part, so only the direct
one runs and must equal the oracle's field of the same rules up to rounding: 1e-11
of the norm (float64 sums of some 1e4 terms, times the near-singular terms'
size).  The expansion's truncation is at most of ratio 1/2 per order at eta = 2:
4 x 2^-(p + 1) of the norm."""
import numpy as np
import pytest

from gpu_util import Plan, rel_l2
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu

XS = np.array([0.1, 0.05, -0.1])


def _setup(m, k, **prm):
    P = Plan(m, bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE, k, **prm)
    phi, ce = I.helmholtz_point_source(m, XS, k) if k else I.point_source(m, XS)
    chi = np.zeros(P.n_chi, ce.dtype)
    chi[P.chi_idx.reshape(-1)] = ce.reshape(-1)
    return P, phi, chi


def _field(P, phi, chi, pts):
    t = P.torch
    xd = t.tensor(pts, device="cuda", dtype=t.float64)
    ud = t.full((len(pts),), float("nan"), device="cuda", dtype=t.complex128 if P.complex else t.float64)
    bem.bem_field(P.plan, P._dev(phi), P._dev(chi), xd, ud)
    t.cuda.synchronize()
    assert bem.bem_plan_device_status(P.plan) == 0
    return ud.cpu().numpy()


def _shell(n, radii, seed=3):
    d = np.random.default_rng(seed).standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return d * np.resize(radii, n)[:, None]


@pytest.mark.parametrize("k", [0.0, 3.0])
@pytest.mark.parametrize("depth,npe,n", [(0, 3, 1), (1, 6, 5), (6, 3, 33), (10, 6, 14)])
def test_direct_part(oracle_lib, k, depth, npe, n):
    m = I.geodesic(4, I.TRI3 if npe == 3 else I.TRI6, axes=(1.0, 0.7, 1.3))
    P, phi, chi = _setup(m, k, p=4, leaf_size=4000, max_subdiv=depth)
    pts = _shell(n, (1.31, 1.45, 2.0)) * [1.0, 0.7, 1.3]
    pts[0] = m.nodes[5] * 1.0005                     # next to a node: every level of subdivision
    st = oracle_lib.Settings(maxdepth=depth)
    ref = oracle_lib.field(m.nodes, m.elems, P.chi_idx, phi, chi, pts, bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE, k, st)
    assert rel_l2(_field(P, phi, chi, pts), ref if k else ref.real) < 1e-11
    P.close()


@pytest.mark.parametrize("p", [1, 2, 3, 9, 14, 20])
@pytest.mark.parametrize("precision", [bem.BEM_F64, bem.BEM_MIXED])
def test_orders(oracle_lib, p, precision):
    m = I.icosphere(2, I.TRI6)
    P, phi, chi = _setup(m, 0.0, p=p, leaf_size=8, eta=2.0, precision=precision)
    pts = _shell(61, (1.1, 2.0, 40.0))
    ref = oracle_lib.field(m.nodes, m.elems, P.chi_idx, phi, chi, pts).real
    assert rel_l2(_field(P, phi, chi, pts), ref) < 4 * 2.0 ** -(p + 1) + (0 if precision == bem.BEM_F64 else 2e-6)
    P.close()


@pytest.mark.parametrize("k", [0.0, 1.5])
def test_level_orders_and_deep_tree(oracle_lib, k):
    m = I.icosphere(3)
    P, phi, chi = _setup(m, k, p=16, p_min=12, leaf_size=2, eta=2.0)
    pts = _shell(101, (1.05, 1.5, 3.0))
    ref = oracle_lib.field(m.nodes, m.elems, P.chi_idx, phi, chi, pts, bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE, k)
    assert rel_l2(_field(P, phi, chi, pts), ref if k else ref.real) < 4 * 2.0 ** -13
    assert _field(P, phi, chi, pts[:0]).size == 0
    P.close()
