"""The kernel instances that only CG iterations run (a single operator
application has its own), element by element: the strain after one, two and
three iterations against the oracle's CG iterates, for every operator form and
every row tile and thread variant of the first and the last pass, two load
cases together.

Bars, of the fluctuation's maximum: FP64 1e-11 (three applications of an
operator that is exact to 1e-12).  FP32 1e-4: an application inside the CG is
exact to about 1e-5 (differences of the displacement along the longest axis of
1024 voxels; 2e-5 is the bar of the operator tests), and three of them, with the
step lengths formed from them, enter the third iterate.  A wrong row, shift or
component changes the field by its own size.
"""
import numpy as np
import pytest

from oracle.fe_projection import Problem
from tests.gpu_util import lognormal, require_gpu

pytestmark = pytest.mark.gpu

GRIDS = [(16, 16), (32, 64), (64, 32), (256, 16), (512, 16), (1024, 16), (16, 1024),
         (16, 16, 16), (32, 16, 64), (64, 32, 16), (128, 16, 16), (256, 16, 16), (16, 256, 16), (16, 16, 256)]
LOADS = (0, 2)


def _iterates(n, steps):
    P = Problem(n, lognormal(n, 191), 0.3, length=(1.0, 0.8, 1.1)[: len(n)])
    out = []
    for l in LOADS:
        cg = P.cg(np.eye(P.ns)[l])
        out.append([next(cg)[0].copy() for _ in range(steps + 1)][1:])
    return P, out


@pytest.mark.parametrize("prec,bar", [("fp64", 1e-11), ("mixed", 1e-4)])
@pytest.mark.parametrize("n", GRIDS)
def test_iterates(n, prec, bar):
    require_gpu()
    from paper_2105_03297_gb300 import RVE, _rve
    P, want = _iterates(n, 3)
    mixed = prec == "mixed"
    va = [0] if n[0] < 64 else [0, 1, 2, 3, 4]
    if mixed and ((len(n) == 2 and n[0] >= 512) or (len(n) == 3 and n[0] >= 128)):
        va.append(5)
    scheds = [(a, 0) for a in va] + ([(0, 1), (0, 2)] if n[0] >= 64 else [])
    Em = np.eye(P.ns)[list(LOADS)]
    for form in ("stress", "factored", "nodal"):
        for sched in scheds if form == "stress" else scheds[-3:]:
            with RVE(n, precision=prec, length=P.length) as r:
                r.set_operator_form(form)
                r.set_schedule(*sched, 0, 0)
                r.set_material(P.E, 0.3)
                for k in (1, 2, 3):
                    code, info = r.solve(Em, rel_tol=1e-14, max_iter=k)
                    assert code == _rve.RVE_ERR_NOT_CONVERGED and [i["iterations"] for i in info] == [k, k], info
                    for l, load in enumerate(LOADS):
                        x = want[l][k - 1]
                        got = r.get_strain(l).reshape(x.shape) - P.broadcast_macro(np.eye(P.ns)[load])
                        assert np.abs(got - x).max() <= bar * np.abs(x).max(), (form, sched, k, l)
