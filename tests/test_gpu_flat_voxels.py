"""Mixed-precision solves on voxels a thousand times as long as they are thick:
the CG vectors have to stay strains of one nodal field, in FP32 as well, or CG
stalls above its tolerance (a node value that two blocks round differently
leaves an incompatible strain of about 2^-24 |w| / h).  Every operator form
against the FP64 handle: convergence, C_eff's column to 1e-9, and no more than
twice the FP64 iterations (each of the three to five refinement steps of the
mixed solve starts a new CG)."""
import numpy as np
import pytest

from tests.gpu_util import lognormal, rel_max, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(32, 32, 32), (64, 16, 32), (16, 64, 16), (64, 64)])
@pytest.mark.parametrize("thin", [0, 1, 2])
def test_flat_voxels(n, thin):
    require_gpu()
    from paper_2105_03297_gb300 import RVE
    if thin >= len(n):
        pytest.skip("two axes")
    # 1 : 1000 between the voxel sizes along `thin` and along the others
    length = [v / 64 for v in n]
    length[thin] *= 1e-3
    E = lognormal(n, 181)

    def solve(prec, form, sched=None):
        with RVE(n, precision=prec, length=length) as r:
            r.set_operator_form(form)
            if sched:
                r.set_schedule(*sched)
            r.set_material(E, 0.3)
            code, info = r.solve(np.eye(r.ns)[:2], rel_tol=1e-10, max_iter=3000)
            assert code == 0, (prec, form, sched, info)
            return r.mean_stress(), max(i["iterations"] for i in info)

    ref, its = solve("fp64", "stress")
    rows = ((0, 0, 0, 0), (1, 1, 0, 0), (2, 2, 0, 0))   # every row tile of the first and last pass
    for form, scheds in (("stress", rows), ("factored", rows[:1]), ("nodal", rows[:1])):
        for sched in scheds:
            S, i = solve("mixed", form, sched)
            assert rel_max(S, ref) < 1e-9, (form, sched)
            assert i <= 2 * its, (form, sched)
