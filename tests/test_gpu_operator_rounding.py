"""Rounding of the FP32 operator on cells of any voxel shape: the 2-norm of the
error of q = G C p on white noise, with inputs that are exact in FP32, against
the FP64 oracle.  Two transforms of up to 2^20 points, each of whose about 20
radix-2 stages adds an independent relative error of about half a unit
roundoff (2^-24), and a few products give some sqrt(40) / 2 + 1 = 4 unit
roundoffs; the bar is twice that, 5e-7, on every grid: neither the grid's nor
the voxel's aspect ratio enters.
"""
import numpy as np
import pytest

from oracle.fe_projection import Problem
from tests.gpu_util import lognormal, require_gpu

pytestmark = pytest.mark.gpu

BAR = 8 * 2.0 ** -24
GRIDS = [(16, 16), (64, 64), (1024, 16), (16, 1024), (1024, 64), (512, 32), (256, 16), (16, 256),
         (16, 16, 16), (256, 16, 16), (16, 256, 16), (16, 16, 256), (64, 32, 16), (128, 16, 64)]


def _case(n):
    E = lognormal(n, 171).astype(np.float32).astype(np.float64)
    P = Problem(n, E, 0.25)
    p = np.random.default_rng(172).standard_normal((P.m,) + E.shape).astype(np.float32)
    return P, E, p, P.operator(p.astype(np.float64)), P.project(p.astype(np.float64))


def _error(q, ref):
    return np.linalg.norm(np.asarray(q, np.float64).ravel() - ref.ravel()) / np.linalg.norm(ref)


@pytest.mark.parametrize("n", GRIDS)
def test_operator(n):
    require_gpu()
    from paper_2105_03297_gb300 import RVE
    P, E, p, ref, bare = _case(n)
    with RVE(n, precision="mixed") as r:
        r.set_material(E, 0.25)
        assert _error(r.apply_operator(p.reshape(P.m, -1)), ref) <= BAR
        assert _error(r.apply_operator(p.reshape(P.m, -1), material=False), bare) <= BAR


@pytest.mark.parametrize("n", [(16, 16), (256, 16), (16, 256), (256, 256)])
def test_operator_without_a_handle(n):
    require_gpu()
    import ctypes as C
    import torch
    from paper_2105_03297_gb300 import _rve
    P, E, p, ref, bare = _case(n)
    Ed, pd = (torch.tensor(v.astype(np.float32).ravel(), device="cuda") for v in (E, p))
    q = torch.empty_like(pd)
    for material, want in ((1, ref), (0, bare)):
        assert 0 == _rve.load().rve_apply_operator_2d_static(
            (C.c_int64 * 2)(*n), None, C.c_void_p(Ed.data_ptr()), 0.25, C.c_void_p(pd.data_ptr()),
            C.c_void_p(q.data_ptr()), material, C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert _error(q.cpu().numpy(), want) <= BAR
