"""Device tensors that the library reads and writes in place: moduli checked and
converted on the device, and the operator's p and q.  The same kernels run on
the same values whichever way the data came, so every comparison is exact."""
import numpy as np
import pytest

from tests.gpu_util import lognormal, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n", [(16, 16), (64, 32)])
def test_device_moduli(n, dtype, prec):
    import torch
    from paper_2105_03297_gb300 import RVE, RveError
    E = lognormal(n, 141).astype(dtype)
    Ed = torch.tensor(E, device="cuda")
    p = np.random.default_rng(142).standard_normal((6, E.size))
    p = p.astype(np.float64 if prec == "fp64" else np.float32)
    with RVE(n, precision=prec) as r:
        r.set_material(E, 0.3)
        ref = r.apply_operator(p)
        r.set_material(2 * E, 0.3)
        r.set_material(Ed, 0.3)
        assert np.array_equal(r.apply_operator(p), ref)
        for where, value in ((0, np.nan), (-1, np.inf), (E.size // 2, -1.0), (slice(None), 0.0)):
            bad = 3 * Ed
            bad.view(-1)[where] = value
            with pytest.raises(RveError):
                r.set_material(bad, 0.3)
            assert np.array_equal(r.apply_operator(p), ref), value   # the earlier material stays
        off = torch.empty(E.size + 1, dtype=Ed.dtype, device="cuda")[1:]   # not 16-byte aligned
        off.copy_(Ed.view(-1))
        r.set_material(off, 0.3)
        assert np.array_equal(r.apply_operator(p), ref)


@pytest.mark.parametrize("own_stream", [False, True])
def test_device_moduli_written_on_the_default_stream(own_stream):
    """Moduli that are still being computed on the default stream when
    set_material is called, on a handle of the default stream and on one of a
    stream that does not wait for it."""
    import torch
    from paper_2105_03297_gb300 import RVE
    n = (64, 64)
    E = lognormal(n, 150)
    p = np.random.default_rng(151).standard_normal((6, E.size))
    a = torch.full((4096, 4096), 1.0 / 4096, device="cuda")
    b, Ed = torch.empty_like(a), torch.ones(E.shape, dtype=torch.float64, device="cuda")
    Eh = torch.tensor(E, device="cuda")
    side = torch.cuda.Stream()   # non-blocking
    with RVE(n, stream=side.cuda_stream if own_stream else None) as r:
        r.set_material(E, 0.3)
        ref = r.apply_operator(p)
        torch.mm(a, a, out=b)
        torch.cuda.synchronize()
        for _ in range(60):   # some milliseconds of queued work
            torch.mm(a, a, out=b)
        Ed.copy_(Eh)
        r.set_material(Ed, 0.3)
        assert np.array_equal(r.apply_operator(p), ref)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [(32, 16), (16, 16, 16)])
def test_operator_on_device_tensors(n, prec):
    import torch
    from paper_2105_03297_gb300 import RVE
    E = lognormal(n, 143)
    m = 6 if len(n) == 2 else 36
    dt = np.float64 if prec == "fp64" else np.float32
    p = np.random.default_rng(144).standard_normal((m, E.size)).astype(dt)
    with RVE(n, precision=prec) as r:
        r.set_material(E, 0.3)
        ref = r.apply_operator(p)
        pd = torch.tensor(p, device="cuda")
        q = r.apply_operator(pd)
        assert np.array_equal(q.cpu().numpy(), ref) and np.array_equal(pd.cpu().numpy(), p)
        wide = torch.empty(2, p.size + 1, dtype=pd.dtype, device="cuda")
        a, b = wide[0, 1:].view(p.shape), wide[1, :-1].view(p.shape)   # of odd alignment
        a.copy_(pd)
        assert np.array_equal(r.apply_operator(a, out=b).cpu().numpy(), ref)
        assert np.array_equal(r.apply_operator(pd, out=a).cpu().numpy(), ref)
        r.apply_operator(pd, out=pd)   # in place
        assert np.array_equal(pd.cpu().numpy(), ref)


@pytest.mark.parametrize("n", [(16, 16), (64, 256)])
def test_static_operator_under_capture(n):
    """A captured call replays on new contents of its buffers like an eager call
    (its three launches are dependent launches, in the graph as on the stream)."""
    import ctypes as C
    import torch
    from paper_2105_03297_gb300 import _rve
    lib = _rve.load()
    E = torch.tensor(lognormal(n, 145).astype(np.float32), device="cuda").view(-1)
    p = torch.empty(6, n[0] * n[1], device="cuda")
    q, ref = torch.empty_like(p), torch.empty_like(p)

    def call(out, stream):
        assert 0 == lib.rve_apply_operator_2d_static(
            (C.c_int64 * 2)(*n), None, C.c_void_p(E.data_ptr()), 0.3, C.c_void_p(p.data_ptr()),
            C.c_void_p(out.data_ptr()), 1, C.c_void_p(stream.cuda_stream))

    call(ref, torch.cuda.current_stream())   # set-up, before the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call(q, torch.cuda.current_stream())
    for seed in (146, 147):
        p.copy_(torch.tensor(np.random.default_rng(seed).standard_normal(p.shape).astype(np.float32)))
        g.replay()
        call(ref, torch.cuda.current_stream())   # same stream: after the replay
        torch.cuda.synchronize()
        assert torch.equal(q, ref) and bool((q != 0).any())


@pytest.mark.parametrize("n", [(16, 16), (256, 64)])
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_static_operator_on_any_element_alignment(n, shift):
    """E, p and q of the entry point without a handle may start at any float,
    and q may be p: the same bits as on aligned fields, and nothing outside."""
    import ctypes as C
    import torch
    from paper_2105_03297_gb300 import _rve
    lib = _rve.load()
    N = n[0] * n[1]
    E = torch.tensor(lognormal(n, 148).astype(np.float32), device="cuda").view(-1)
    p = torch.tensor(np.random.default_rng(149).standard_normal(6 * N).astype(np.float32), device="cuda")
    q = torch.empty_like(p)

    def call(E, p, q):
        assert 0 == lib.rve_apply_operator_2d_static(
            (C.c_int64 * 2)(*n), None, C.c_void_p(E.data_ptr()), 0.3, C.c_void_p(p.data_ptr()),
            C.c_void_p(q.data_ptr()), 1, C.c_void_p(torch.cuda.current_stream().cuda_stream))

    def shifted(t):
        w = torch.full((t.numel() + 8,), 7.0, device="cuda")
        v = w[shift:shift + t.numel()]
        v.copy_(t)
        return w, v

    call(E, p, q)
    (_, Es), (pw, ps), (qw, qs) = shifted(E), shifted(p), shifted(torch.zeros_like(p))
    call(Es, ps, qs)
    assert torch.equal(qs, q) and torch.equal(ps, p)
    call(Es, ps, ps)
    assert torch.equal(ps, q)
    for w in (pw, qw):
        assert bool((w[:shift] == 7).all()) and bool((w[shift + 6 * N:] == 7).all())


CAPTURED_FIRST = r"""
import ctypes as C, json, sys
import torch
sys.path.insert(0, sys.argv[1])
from paper_2105_03297_gb300 import RVE, _rve
n = (64, 32)
g = torch.Generator(device="cuda").manual_seed(5)
E = torch.rand(n[0] * n[1], device="cuda", generator=g) + 0.5
p = torch.randn(6, n[0] * n[1], device="cuda", generator=g)
q, captured = torch.zeros_like(p), torch.zeros_like(p)
lib = _rve.load()
with RVE(n, precision="mixed") as r:    # also loads the library's device code
    r.set_material(E, 0.3)
    ref = r.apply_operator(p)

def call(out):
    return lib.rve_apply_operator_2d_static((C.c_int64 * 2)(*n), None, C.c_void_p(E.data_ptr()), 0.3,
                                            C.c_void_p(p.data_ptr()), C.c_void_p(out.data_ptr()), 1,
                                            C.c_void_p(torch.cuda.current_stream().cuda_stream))

graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph, capture_error_mode="relaxed"):
    rc1 = call(captured)
rc2 = call(q)                           # the captured call has not run
torch.cuda.synchronize()
eager = q.clone()
graph.replay()
torch.cuda.synchronize()
# (the tables of the two entry points may differ in the last bit)
print(json.dumps([rc1, rc2, float((eager - ref).norm() / ref.norm()) < 5e-7, torch.equal(captured, eager)]))
"""


def test_static_operator_whose_first_call_is_captured():
    """In a process of its own: a first call that is only captured leaves the
    set-up of the tables to the next call, and carries its own when replayed."""
    import json
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    res = subprocess.run([sys.executable, "-c", CAPTURED_FIRST, root], capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stderr[-2000:]
    assert json.loads(res.stdout.strip().splitlines()[-1]) == [0, 0, True, True]
