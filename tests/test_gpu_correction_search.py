"""The special-pair search where its float32 tests cannot decide: meshes far
from the origin (the rounding margin grows past the radii and the float64
classification takes every element), radii below and above an element's own
extent, no special radius at all, and nodes with more pairs than the search
keeps.  The pairs' entries (their columns in order, too) against the oracle's:
integers, so exactly."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from gpu_util import Plan
from paper_0908_0673_gb300 import bem, inputs as I

pytestmark = pytest.mark.gpu

MESHES = {
    "sphere-tri3": lambda: I.icosphere(2),
    "cube-tri6": lambda: I.cube(4, I.TRI6),
}


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("shift", [0.0, 30.0, 1e5])
@pytest.mark.parametrize("tau", [0.0, 0.6, 2.0, 9.0])
@pytest.mark.parametrize("precision", [bem.BEM_F64, bem.BEM_MIXED])
def test_pairs(name, shift, tau, precision):
    m = MESHES[name]()
    m = dataclasses.replace(m, nodes=np.ascontiguousarray(m.nodes + np.array([shift, -0.5 * shift, 0.25 * shift])))
    P = Plan(m, p=4, leaf_size=32, precision=precision, tau_near=tau, max_subdiv=1)
    st = O.Settings(tau=tau, maxdepth=1)
    ref = O.correction(m.nodes, m.elems, P.chi_idx, st=st)
    got = bem.bem_plan_export_correction(P.plan)
    for part, cols in (("D", ref["col_phi"]), ("S", ref["col_chi"])):
        key = lambda r, c: np.sort(r.astype(np.int64) * 10 ** 7 + c)
        assert np.array_equal(key(got["row" + part], got["col" + part]), key(ref["row"], cols)), part
    P.close()
