"""The finite-element passes on the D nodal components (B^H and B taken as
differences along y and z, the y and z transforms of three or two components)
against the FP64 oracle, at the edges of their tiles: the shortest axes, rows
of one warp and of several, one and several z chunks, grids smaller than a
tile, voxels of unequal size, and every row tile of the last pass.  Operator
q = G C p and bare projection q = G p, FP64 to 1e-12 and FP32 to 2e-5 of the
field maximum.
"""
import numpy as np
import pytest

from oracle.fe_projection import Problem
from tests.gpu_util import lognormal, require_gpu

pytestmark = pytest.mark.gpu

GRIDS = [(16, 16), (16, 1024), (1024, 16), (32, 64), (512, 32),
         (16, 16, 16), (16, 32, 64), (64, 16, 32), (32, 64, 16), (128, 16, 16), (16, 128, 32)]


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 2e-5)])
def test_operator_and_projection(n, prec, tol):
    require_gpu()
    from paper_2105_03297_gb300 import RVE
    length = (1.0, 0.7, 1.3)[: len(n)]
    E = lognormal(n, 131)
    P = Problem(n, E, 0.3, length=length)
    p = np.random.default_rng(132).standard_normal((P.m,) + E.shape)
    if prec == "mixed":
        p = p.astype(np.float32).astype(np.float64)
    ref, bare = P.operator(p), P.project(p)
    variants = 1 if n[0] < 64 else 5 if (len(n) == 3 and prec == "mixed" and n[0] >= 128) else 3
    with RVE(n, precision=prec, length=length) as r:
        r.set_material(E, 0.3)
        for v in range(variants):
            r.set_schedule(0, v)
            q = r.apply_operator(p.reshape(P.m, -1)).reshape(ref.shape)
            assert np.abs(q - ref).max() <= tol * np.abs(ref).max(), v
            q = r.apply_operator(p.reshape(P.m, -1), material=False).reshape(ref.shape)
            assert np.abs(q - bare).max() <= tol * np.abs(bare).max(), v
