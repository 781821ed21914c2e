"""The float32 near field at the edges of its passes, clusters and ranges, on
meshes of one box (no far field), against the dense oracle.  Tolerance: the
mixed product's stated bar, 2e-6 of the norm; a Helmholtz phase k r adds
2^-22 k r (its rounding and its arguments', float32)."""
import numpy as np
import pytest

import oracle as O
from gpu_util import Plan, rel_l2
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu

MESHES = {
    "12-nodes": (lambda: I.icosphere(0), dict(p=8, leaf_size=64)),                       # 2 groups, a cluster of 8
    "98-nodes-tri6": (lambda: I.cube(2, I.TRI6, grade=0.0), dict(p=8, leaf_size=128)),   # 64 + 34 targets
    "162-nodes": (lambda: I.icosphere(2), dict(p=8, leaf_size=256)),                     # 2 x 64 + 34
    "deep": (lambda: I.icosphere(3), dict(p=16, leaf_size=3, eta=8.0)),                  # 522 near entries: several chunks
}


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("k", [0.0, 2.0])
def test_all_near_equals_dense(name, k):
    make, prm = MESHES[name]
    m = make()
    green = bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE
    P = Plan(m, green, k, precision=bem.BEM_MIXED, **prm)
    A, B, _ = O.operators(m.nodes, m.elems, P.chi_idx, P.n_chi, green=green, k=k)
    for op, M in ((bem.BEM_OP_A, A), (bem.BEM_OP_B, B)):
        x = I.random_vector(M.shape[1], 3, bool(k))
        assert rel_l2(P.matvec(op, x), M @ x) < 2e-6
    P.close()


@pytest.mark.parametrize("k", [1e-4, 40.0, 1500.0, 1700.0])
def test_phase_range(k):
    """From a phase far below one table step to either side of the table's limit."""
    m = I.icosphere(1)
    P = Plan(m, bem.BEM_HELMHOLTZ, k, p=4, leaf_size=64, precision=bem.BEM_MIXED)
    A, B, _ = O.operators(m.nodes, m.elems, P.chi_idx, P.n_chi, green=bem.BEM_HELMHOLTZ, k=k)
    for op, M in ((bem.BEM_OP_A, A), (bem.BEM_OP_B, B)):
        x = I.random_vector(M.shape[1], 4, True)
        assert rel_l2(P.matvec(op, x), M @ x) < 2e-6 + 2.0 ** -22 * 2 * k
    P.close()
