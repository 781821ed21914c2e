"""The float64 near field in float32 pairs at the edges of its tiles and ranges.

Meshes that fit one box have no far field, and at eta = 8, p = 16 the little
there is has a truncation error of 8^-17, so the product must equal the dense
oracle's up to rounding.  Tolerance: a pair's
relative error is at most about 2^-44 (48-bit words through some twenty
dependent operations), a singular or near-singular pair's regular value, which
the stored correction takes out again, is at most a few hundred times its
node's result, and the two sides' float64 sums differ by some 1e-13: 1e-11 of
the result's norm.  A Helmholtz phase k r carries 2^-46 k r more.
"""
import numpy as np
import pytest

import oracle as O
from gpu_util import Plan, rel_l2
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu

MESHES = {
    "12-nodes": (lambda: I.icosphere(0), dict(p=8, leaf_size=64)),                   # one item, 12 of 32 targets
    "42-nodes": (lambda: I.icosphere(1), dict(p=8, leaf_size=64)),                   # 32 + 10 targets
    "98-nodes-tri6": (lambda: I.cube(2, I.TRI6, grade=0.0), dict(p=8, leaf_size=128)),  # 3 x 32 + 2
    "deep": (lambda: I.icosphere(3), dict(p=16, leaf_size=3, eta=8.0)),              # 522 near entries: several chunks
}


def _dense(m, P, green=bem.BEM_LAPLACE, k=0.0):
    A, B, _ = O.operators(m.nodes, m.elems, P.chi_idx, P.n_chi, green=green, k=k)
    return A, B


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("k", [0.0, 2.0])
def test_all_near_equals_dense(name, k):
    make, prm = MESHES[name]
    m = make()
    green = bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE
    P = Plan(m, green, k, **prm)
    if name == "deep":
        assert np.diff(bem.bem_plan_export_tree(P.plan)["near_ptr"]).max() > 256
    A, B = _dense(m, P, green, k)
    for op, M, n in ((bem.BEM_OP_A, A, P.n_phi), (bem.BEM_OP_B, B, P.n_chi)):
        x = I.random_vector(n, 3, bool(k))
        assert rel_l2(P.matvec(op, x), M @ x) < 1e-11
    P.close()


@pytest.mark.parametrize("k", [300.0, 500.0])
def test_phase_table_limit(k):
    """Below the limit the table form runs, above it the float64 kernel."""
    m = I.icosphere(1)
    P = Plan(m, bem.BEM_HELMHOLTZ, k, p=4, leaf_size=64)
    A, B = _dense(m, P, bem.BEM_HELMHOLTZ, k)
    for op, M in ((bem.BEM_OP_A, A), (bem.BEM_OP_B, B)):
        x = I.random_vector(M.shape[1], 4, True)
        assert rel_l2(P.matvec(op, x), M @ x) < 1e-11 + 2.0 ** -46 * 2 * k
    P.close()


@pytest.mark.parametrize("s", [2.0 ** -70, 2.0 ** 70])
def test_scale_of_the_body(s):
    """Op A does not change with the body's size, op B goes with it (exact powers of two)."""
    m, big = I.icosphere(1), I.icosphere(1)
    big.nodes = big.nodes * s
    P, Q = Plan(m, p=8, leaf_size=64), Plan(big, p=8, leaf_size=64)
    x = I.random_vector(P.n_phi, 5)
    assert rel_l2(Q.matvec(bem.BEM_OP_A, x), P.matvec(bem.BEM_OP_A, x)) < 1e-13
    x = I.random_vector(P.n_chi, 5)
    assert rel_l2(Q.matvec(bem.BEM_OP_B, x) / s, P.matvec(bem.BEM_OP_B, x)) < 1e-13
    P.close()
    Q.close()


@pytest.mark.parametrize("k", [0.0, 2.0])
def test_scale_and_spread_of_the_vector(k):
    m = I.icosphere(2)
    P = Plan(m, bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE, k, p=8, leaf_size=16)
    x = I.random_vector(P.n_phi, 6, bool(k))
    y = P.matvec(bem.BEM_OP_A, x)
    for s in (2.0 ** -900, 2.0 ** 900):
        assert rel_l2(P.matvec(bem.BEM_OP_A, x * s) / s, y) < 1e-13
    z = P.matvec(bem.BEM_OP_A, np.zeros_like(x))
    assert np.all(z == 0)
    a, b = x.copy(), x.copy()
    a[::2] *= 1e-40                                # both halves of a sum of very different magnitudes
    b[::2] = 0
    b[1::2] = x[1::2]
    c = x.copy()
    c[1::2] = 0
    ref = P.matvec(bem.BEM_OP_A, b) + 1e-40 * P.matvec(bem.BEM_OP_A, c)
    assert rel_l2(P.matvec(bem.BEM_OP_A, a), ref) < 1e-13
    x[7] = np.nan
    assert not np.isfinite(P.matvec(bem.BEM_OP_A, x)).any()
    P.close()
