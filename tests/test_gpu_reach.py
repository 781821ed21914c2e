"""float64 plans of meshes with fine detail beside large elements.

An element belongs to the leaf of its first node.  Here three triangles of an
icosphere are each replaced by a fan of 81 tiny triangles joined to the corners
by long ones whose first node lies on the fan's ring, so that leaves of level 10
to 15 own quadrature points 90 to 2,900 edges from their centres: powers of such
an offset / edge pass float32's range at the diagonal's order 16, and leading
moments lie far below the highest ones.

Tolerances: products against the oracle's fast product on the same tree (same
truncation) 2e-9: coordinates carry 2^-53 of the body's size and the quadrature
points nearest a ring node are a tenth of a 7.8e-6 side away, a few 1e-10 of an
entry, and 1e-9 is the bar of the other parity tests; the diagonal against the
dense row sums 5e-8, its stated accuracy."""
import functools

import numpy as np
import pytest

import oracle as O

from gpu_util import Plan, rel_l2
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu


def ringed(rad, n=81):
    """An icosphere of 320 triangles, every 107th replaced by a fan of radius rad."""
    m = I.icosphere(2)
    cut = set(range(0, m.n_elems, 107))
    nodes, tri, N = [m.nodes], [t for i, t in enumerate(m.elems) if i not in cut], len(m.nodes)
    for i in cut:
        corner = m.elems[i]
        P = m.nodes[corner]
        cen = P.mean(0)
        u = (P[0] - cen) / np.linalg.norm(P[0] - cen)
        w = np.cross(P[1] - P[0], P[2] - P[0])
        v = np.cross(w / np.linalg.norm(w), u)
        th = 2 * np.pi * np.arange(n) / n
        nodes += [cen + rad * (np.outer(np.cos(th), u) + np.outer(np.sin(th), v)), cen[None]]
        at = np.arctan2((P - cen) @ v, (P - cen) @ u)
        near = [int(np.argmin(np.abs((t + np.pi / n - at + np.pi) % (2 * np.pi) - np.pi))) for t in th]
        for j in range(n):
            q, r, k = N + j, N + (j + 1) % n, near[(j + 1) % n]
            tri += [[q, r, N + n], [q, corner[near[j]], r]]
            if k != near[j]:
                tri.append([r, corner[near[j]], corner[k]])
        N += n + 1
    m.nodes, m.elems = np.vstack(nodes), np.array(tri, np.int32)
    return m


@functools.lru_cache(maxsize=None)
def _reference(rad, k):
    m = ringed(rad)
    idx, n = O.chi_index(m.nodes, m.elems)
    return (m, idx, O.assemble(m.nodes, m.elems, idx, n)[2],
            O.correction(m.nodes, m.elems, idx, O.HELMHOLTZ if k else O.LAPLACE, k))


@pytest.mark.parametrize("k", [0.0, 2.0])
@pytest.mark.parametrize("rad,leaf,p", [(1e-3, 64, 8), (1e-3, 16, 20), (1e-4, 64, 16), (1e-4, 16, 10), (1e-4, 64, 20)])
def test_points_far_beyond_the_leaf(oracle_lib, rad, leaf, p, k):
    m, idx, d0, corr = _reference(rad, k)
    green = bem.BEM_HELMHOLTZ if k else bem.BEM_LAPLACE
    T = oracle_lib.Tree(m.nodes, m.elems, B=leaf, eta=2.0)
    reach = T.radius * 2.0 ** T.level / T.side
    assert reach[T.leaf == 1].max() > 20 and reach[T.inter_idx].max() > 8     # leaves, and boxes that are read
    P = Plan(m, green, k, p=p, leaf_size=leaf, eta=2.0)
    try:
        diag = bem.bem_plan_diagonal(P.plan, P.n_phi)
        assert np.array_equal(idx, P.chi_idx)
        assert np.abs(diag - 1.0 - d0).max() < 5e-8
        for op, n in ((bem.BEM_OP_A, P.n_phi), (bem.BEM_OP_B, P.n_chi)):
            x = I.random_vector(n, 60 + op, bool(k))
            ref = oracle_lib.fmm_apply(T, P.chi_idx, op, x, diag - 1.0, corr, p, green, k)
            assert rel_l2(P.matvec(op, x), ref if k else ref.real) < 2e-9, op
    finally:
        P.close()
