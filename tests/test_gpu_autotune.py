"""The autotuner times the kernels that a handle runs: its choices are kept per
operator form and derivative, and a handle that changes them is tuned again.
The grids are used by no other test, so nothing of theirs is cached yet."""
import numpy as np
import pytest

from tests.gpu_util import lognormal, require_gpu

pytestmark = pytest.mark.gpu


def _tuned(r, L):
    """The schedule and the candidates that were timed by a solve of L load cases."""
    code, info = r.solve(np.eye(r.ns)[:L], rel_tol=1e-6, max_iter=2000)
    assert code == 0, info
    var, ms = r.schedule()
    return var, [[v for v, t in enumerate(row) if t > 0] for row in ms]


def test_choices_of_one_derivative_are_not_anothers():
    require_gpu()
    from paper_2105_03297_gb300 import RVE
    n, E = (64, 256), lognormal((64, 256), 161)
    with RVE(n) as a, RVE(n) as b, RVE(n) as c:
        for r in (a, b, c):
            r.set_material(E, 0.3)
        a.set_derivative("fourier")
        assert _tuned(a, 2)[1][0] == [0, 1, 2, 3, 4]
        var, timed = _tuned(b, 2)
        assert timed[0] == [0, 1, 2, 3, 4]            # the force pass's own candidates
        c.set_derivative("fourier")
        assert _tuned(c, 2) == (a.schedule()[0], [[], [], [], []])   # from the cache
        c.set_derivative("fe")
        assert c.schedule()[0] == [-1] * 4
        assert _tuned(c, 2)[0] == var
        c.set_schedule(1, 1)                          # the caller's entries stay
        c.set_derivative("fourier")
        assert c.schedule()[0][:2] == [1, 1]


def test_choices_of_one_form_are_not_anothers():
    require_gpu()
    from paper_2105_03297_gb300 import RVE
    n, E = (128, 16, 64), lognormal((128, 16, 64), 162)
    timed = {}
    for form in ("factored", "nodal", "stress"):
        with RVE(n, precision="mixed") as r:
            r.set_operator_form(form)
            r.set_material(E, 0.3)
            var, timed[form] = _tuned(r, 2)
            assert form == "stress" or var[0] != 5
    assert timed["factored"][:2] == [[0, 1, 2, 3, 4], [0, 1, 2]]
    assert timed["nodal"][:2] == [[0], [0]]           # its first and last passes have one shape
    assert timed["stress"][:2] == [[0, 1, 2, 3, 4, 5], [0, 1, 2]]
