"""The SIMT M2L, and the float64 P2M before it, at the edges of its row blocks, row chunks, column tail and
image batches: orders 1 to 20, both Green's functions and precisions, against
the oracle's fast product on the same tree (same truncation, so only rounding
differs).  Tolerances: float64 plans 1e-9, the bar of the other parity tests
(48-bit words leave some 1e-13); mixed plans 2e-6, their stated bar."""
import pytest

from gpu_util import Plan, rel_l2
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu


def _check(oracle_lib, m, p, leaf, k, precision, tol, p_min=0):
    green = bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE
    P = Plan(m, green, k, p=p, leaf_size=leaf, eta=2.0, precision=precision, p_min=p_min)
    try:
        assert not P.stats()["m2l_tensor_cores"] and P.stats()["m2l_classes"] > 5
        T = oracle_lib.Tree(m.nodes, m.elems, B=leaf, eta=2.0)
        d0 = bem.bem_plan_diagonal(P.plan, P.n_phi) - 1.0
        corr = oracle_lib.correction(m.nodes, m.elems, P.chi_idx, green, k)
        for op, n in ((bem.BEM_OP_A, P.n_phi), (bem.BEM_OP_B, P.n_chi)):
            x = I.random_vector(n, 50 + op, bool(k))
            ref = oracle_lib.fmm_apply(T, P.chi_idx, op, x, d0, corr, p, green, k)
            e = rel_l2(P.matvec(op, x), ref if k else ref.real)
            assert e < tol, (op, e)
        assert bem.bem_plan_device_status(P.plan) == 0
    finally:
        P.close()


@pytest.mark.parametrize("k", [0.0, 2.0])
@pytest.mark.parametrize("p", [1, 2, 3, 5, 9, 11, 14])
def test_float64_orders(oracle_lib, p, k):
    _check(oracle_lib, I.icosphere(2), p, 4, k, bem.BEM_F64, 1e-9)


@pytest.mark.parametrize("k,p", [(0.0, 13), (0.0, 16), (2.0, 1), (2.0, 4), (2.0, 8), (2.0, 10), (2.0, 15)])
def test_mixed_orders(oracle_lib, p, k):
    """Laplace above the tensor cores' orders, Helmholtz at every kind."""
    _check(oracle_lib, I.icosphere(2), p, 4, k, bem.BEM_MIXED, 2e-6)


@pytest.mark.parametrize("k", [0.0, 2.0])
@pytest.mark.parametrize("p,leaf", [(6, 12), (13, 40)])
def test_large_leaves(oracle_lib, k, p, leaf):
    """Leaves of one and of several P2M rounds (64 points), on both row widths."""
    _check(oracle_lib, I.icosphere(3), p, leaf, k, bem.BEM_F64, 1e-9)


@pytest.mark.parametrize("k", [0.0, 2.0])
def test_images_in_batches(oracle_lib, k):
    """Order 20: 1.8 MB a class (3.7 complex), so the images are built a batch at a time."""
    _check(oracle_lib, I.geodesic(3, I.TRI3, axes=(0.6, 1.0, 1.7)), 20, 3, k, bem.BEM_F64, 1e-9)
