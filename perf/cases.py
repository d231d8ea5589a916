"""The work this package is measured on: solves, batches, gradients and single
operator applications through its public entry points.

``listed()`` gives the cases, ``draw(rng)`` another one of the same ranges,
``prepare(case, seed)`` what a program holds before the call, ``run(state)`` one
pass, ``work(case)`` the bytes and operations a pass cannot do without, and
``exact(case, seed)`` the same outputs in 64 bits from plain torch.

A case is a flat dict: ``do`` names the entry point, ``nx, ny, nz`` the grid (nz
= 1: two dimensions; every axis a power of two, 16..1024 in 2D and 16..256 in
3D), ``precision`` "fp64" or "mixed", ``form`` the order of the operator inside
the CG iterations, ``field`` the kind of microstructure, ``loads`` the number of
unit macroscopic strains solved together and ``tol`` the relative residual.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2105_03297_gb300 import RVE, RVEBatch, _rve
from paper_2105_03297_gb300.autograd import effective_stiffness

NU = 0.3
MAX_ITER = 20000
DEV = "cuda"
F_MACRO = [[1.05, 0.02], [0.0, 0.97]]


def _case(name, do, grid, **more):
    nx, ny, nz = (tuple(grid) + (1,))[:3]
    c = dict(name=name, do=do, nx=nx, ny=ny, nz=nz, precision="mixed", form="stress", field="lognormal", loads=1,
             tol=1e-11)
    c.update(more)
    return c


def listed():
    return [
        # one operator application without a handle, the smallest call there
        # is: a caller's own iteration on a small 2D cell, bound by launches
        _case("static_op_64x64", "static_op", (64, 64)),
        # the operator on a handle in the default precision (FP64), a caller's
        # own solver on a mid-size, non-square 2D cell
        _case("op_fp64_512x256", "operator", (512, 256), precision="fp64"),
        # the same in the fast precision on a 3D cell: 36 strain components
        _case("op_mixed_128x128x128", "operator", (128, 128, 128)),
        # the smallest full solve: a 32 x 32 disc, three load cases, in the
        # default precision; bound by launches and the host's part
        _case("solve_fp64_32x32", "solve", (32, 32), precision="fp64", field="disc", loads=3),
        # the 2D homogenisation of the benchmark: a 1024 x 1024 two-phase field,
        # three load cases
        _case("solve_mixed_1024x1024", "solve", (1024, 1024), field="two_phase", loads=3),
        # 16 RVEs of uneven size (64..512 per side), as a data-set generator
        # sends them
        _case("batch_mixed_16", "batch", (512, 512), field="two_phase", loads=3, count=16),
        # the full tangent of a small 3D cell, six load cases in one solve
        _case("solve_mixed_64x64x64", "solve", (64, 64, 64), loads=6),
        # a large, flat 3D cell in the default operator form, one load case
        _case("solve_mixed_256x256x64", "solve", (256, 256, 64), tol=1e-10),
        # the largest grid, in the form for large cells (nodal state)
        _case("solve_nodal_256x256x256", "solve", (256, 256, 256), form="nodal", tol=1e-10),
        # gradient of an objective of the tangent with respect to every
        # modulus: one step of an optimiser, forward and backward
        _case("gradient_mixed_64x64x64", "gradient", (64, 64, 64), tol=1e-10),
        # the solve in the default precision on a mid-size 2D cell, with the
        # Fourier derivative for comparison runs
        _case("solve_fourier_fp64_256x256", "solve", (256, 256), precision="fp64", field="two_phase", loads=3,
              derivative="fourier", tol=1e-12),
        # finite strain (Newton), one macroscopic deformation
        _case("finite_fp64_256x128", "finite", (256, 128), precision="fp64", tol=1e-10),
    ]


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo, hi)


def _cost(c):
    """Rough relative cost of a drawn case (voxels x load cases x iterations x
    what a voxel costs in its precision and form), to bound what draw() gives."""
    n = c["nx"] * c["ny"] * c["nz"]
    three = c["nz"] > 1
    per = (6.7 if three else 1.1) if c["precision"] == "fp64" else (0.43 if three else 0.09)
    if c["form"] != "stress" and c["precision"] == "mixed":
        per *= 0.3
    its = {"static_op": 1, "operator": 1, "gradient": 2 * 260, "finite": 400}.get(c["do"], 260)
    return n * c["loads"] * per * its * (c.get("count", 1) / 4 if c["do"] == "batch" else 1)


def draw(rng):
    """One more case: the kind by use, each axis a power of two drawn on its own
    (so most grids are not square), the options of that kind."""
    while True:
        do = rng.choice(["static_op", "operator", "operator", "solve", "solve", "solve", "solve", "batch", "gradient",
                         "finite"])
        if do == "static_op":
            c = _case("", do, (_pow2(rng, 4, 8), _pow2(rng, 4, 8)))
        elif do == "operator":
            three = rng.random() < 0.5
            grid = tuple(_pow2(rng, 4, 8 if three else 10) for _ in range(3 if three else 2))
            c = _case("", do, grid, precision=rng.choice(["fp64", "mixed"]))
        elif do == "solve":
            three = rng.random() < 0.6
            precision = rng.choice(["fp64", "mixed", "mixed"])
            grid = tuple(_pow2(rng, 4, (6 if precision == "fp64" else 8) if three else 10) for _ in range(3 if three else 2))
            c = _case("", do, grid, precision=precision, field=rng.choice(["lognormal", "two_phase"]),
                      form=rng.choice(["stress", "stress", "factored", "nodal", "nodal"]),
                      loads=rng.choice([1, 6 if three else 3, rng.randint(1, 6 if three else 3)]))
            if not three and precision == "fp64" and rng.random() < 0.4:
                c.update(form="stress", derivative=rng.choice(["fourier", "forward", "lsq"]), tol=1e-12)
        elif do == "batch":
            c = _case("", do, (512, 512), field="two_phase", loads=3, count=rng.randint(2, 16))
        elif do == "gradient":
            three = rng.random() < 0.6
            grid = tuple(_pow2(rng, 4, 6 if three else 8) for _ in range(3 if three else 2))
            c = _case("", do, grid, loads=6 if three else 3, tol=1e-10)
        else:
            c = _case("", do, (_pow2(rng, 4, 8), _pow2(rng, 4, 8)), precision="fp64", tol=1e-10)
        if _cost(c) <= 0.7 * 4194304 * 0.43 * 260 and c["nx"] * c["ny"] * c["nz"] * c["loads"] <= 4194304:
            del c["name"]
            return c


# ------------------------------------------------------------------ inputs
def _grid(case):
    return (case["nx"], case["ny"]) + ((case["nz"],) if case["nz"] > 1 else ())


def _shape(n):
    return tuple(reversed(n))


def _smooth(noise, sigma):
    """Periodic Gaussian blur of `noise`, sigma in voxels."""
    hat = torch.fft.rfftn(noise)
    dim = noise.dim()
    for ax, size in enumerate(noise.shape):
        f = (torch.fft.rfftfreq if ax == dim - 1 else torch.fft.fftfreq)(size, device=noise.device, dtype=noise.dtype)
        g = torch.exp(-2.0 * (math.pi * f * sigma) ** 2)
        hat = hat * g.reshape([-1 if a == ax else 1 for a in range(dim)])
    return torch.fft.irfftn(hat, s=noise.shape)


def _moduli(n, field, gen):
    """Per-voxel Young's moduli of a seeded microstructure (x fastest)."""
    shape = _shape(n)
    if field == "disc":  # a disc of radius 0.25 +- 0.05 at a random place, 10 times as stiff
        r = 0.25 + 0.05 * (2 * torch.rand(1, generator=gen, device=DEV, dtype=torch.float64) - 1)
        at = torch.rand(len(n), generator=gen, device=DEV, dtype=torch.float64)
        d2 = torch.zeros(shape, device=DEV, dtype=torch.float64)
        for ax, size in enumerate(shape):
            t = ((torch.arange(size, device=DEV, dtype=torch.float64) + 0.5) / size - at[ax] + 0.5) % 1.0 - 0.5
            d2 = d2 + (t * t).reshape([-1 if a == ax else 1 for a in range(len(n))])
        return torch.where(d2 < r * r, 10.0, 1.0).to(torch.float64)
    noise = torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64)
    if field == "lognormal":
        return torch.exp(noise)
    soft = _smooth(noise, 8.0 if len(n) == 2 and max(n) > 128 else 3.0)
    cut = torch.quantile(soft.reshape(-1)[: 1 << 20], 0.5)
    return torch.where(soft > cut, 100.0 if len(n) == 2 else 20.0, 1.0).to(torch.float64)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _batch_sizes(case):
    """Grids of a batch: they belong to the case, the fields to the seed."""
    pick = np.random.default_rng(int(case["count"]))
    pairs = zip(pick.choice([64, 128, 256, 512], case["count"]), pick.choice([1, 1, 2], case["count"]))
    return [(int(s), max(64, int(s) // int(t))) for s, t in pairs]


def _inputs(case, seed):
    """The seeded inputs of a case, on the device (a batch's on the host, where
    its entry point takes them)."""
    n, gen = _grid(case), _gen(seed)
    ns = 3 if len(n) == 2 else 6
    if case["do"] in ("operator", "static_op"):
        dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        return dict(E=_moduli(n, case["field"], gen),
                    p=torch.randn(ns * (2 if len(n) == 2 else 6), math.prod(n), generator=gen, device=DEV, dtype=dtype))
    if case["do"] == "batch":
        sizes = _batch_sizes(case)
        return dict(sizes=sizes, E=[_moduli(s, case["field"], gen).cpu().numpy() for s in sizes])
    if case["do"] == "gradient":
        w = torch.rand(ns, ns, generator=gen, device=DEV, dtype=torch.float64)
        return dict(E=_moduli(n, case["field"], gen), W=w + w.T)
    return dict(E=_moduli(n, case["field"], gen))


def _loads(case):
    return np.eye(6 if case["nz"] > 1 else 3)[: case["loads"]]


def prepare(case, seed):
    st = dict(_inputs(case, seed), case=case)
    n, do = _grid(case), case["do"]
    if do == "batch":
        st["h"] = RVEBatch(st["sizes"], precision=case["precision"], nu=NU)
    elif do == "static_op":
        st["lib"] = _rve.load()
        st["E"] = st["E"].to(torch.float32)
        st["q"] = torch.empty_like(st["p"])
    elif do != "gradient":
        h = st["h"] = RVE(n, precision=case["precision"])
        if case["form"] != "stress":
            h.set_operator_form(case["form"])
        if "derivative" in case:
            h.set_derivative(case["derivative"])
        if do == "finite":
            h.set_kinematics("finite")
        if do == "operator":
            h.set_material(st["E"].reshape(-1), NU)
            st["q"] = torch.empty_like(st["p"])
        if do == "solve":
            st["eps"] = [torch.empty(h.m, h.N, dtype=torch.float64, device=DEV) for _ in range(case["loads"])]
    return st


# --------------------------------------------------------------------- run
def run(st):
    case, do = st["case"], st["case"]["do"]
    if do == "static_op":
        nn = (ctypes.c_int64 * 2)(case["nx"], case["ny"])
        ptr = ctypes.c_void_p
        code = st["lib"].rve_apply_operator_2d_static(nn, None, ptr(st["E"].data_ptr()), NU, ptr(st["p"].data_ptr()),
                                                      ptr(st["q"].data_ptr()), 1,
                                                      ptr(torch.cuda.current_stream().cuda_stream))
        if code:
            raise _rve.RveError(code, "rve_apply_operator_2d_static")
        return st["q"]
    if do == "operator":
        return st["h"].apply_operator(st["p"], out=st["q"])
    if do == "batch":
        for i, E in enumerate(st["E"]):
            st["h"].set_material(i, E)
        st["h"].solve(_loads(case), rel_tol=case["tol"], max_iter=MAX_ITER)
        return np.stack([st["h"].effective_tangent(i) for i in range(len(st["E"]))])
    if do == "gradient":
        E = st["E"].detach().requires_grad_(True)
        C = effective_stiffness(E, NU, precision=case["precision"], rel_tol=case["tol"])
        (C * st["W"]).sum().backward()
        return {"C": C.detach(), "grad": E.grad}
    h = st["h"]
    h.set_material(st["E"].reshape(-1), NU)
    if do == "finite":
        h.solve_finite(np.array([F_MACRO]), rel_tol=case["tol"])
        return {"P": h.mean_piola(), "F": h.get_deformation(0)}
    h.solve(_loads(case), rel_tol=case["tol"], max_iter=MAX_ITER)
    return {"S": h.mean_stress(), "eps": [h.get_strain(l, out=e) for l, e in enumerate(st["eps"])]}


# -------------------------------------------------------------------- work
def _grid_work(n, loads, its, nq):
    """Operations of `its` iterations of the projected solve: per load case the
    real FFTs there and back of the D nodal components and the material law on
    every element (strain, stress, force: about 60 operations each in 2D, 90 in
    3D), which no order of the operator does without."""
    D, N = len(n), math.prod(n)
    return loads * its * (2 * D * 2.5 * N * math.log2(N) + N * nq * (60 if D == 2 else 90))


def work(case):
    n, do = _grid(case), case["do"]
    D, N = len(n), math.prod(n)
    ns, nq = (3, 2) if D == 2 else (6, 6)
    if case.get("derivative") in ("fourier", "forward", "lsq"):
        nq = 1
    if do in ("operator", "static_op"):
        s = 8 if case["precision"] == "fp64" else 4
        return {"bytes": (2 * ns * nq + 1) * N * s, "flops": _grid_work(n, 1, 1, nq)}
    if do == "batch":
        sizes = _batch_sizes(case)
        return {"bytes": sum(8 * a * b for a, b in sizes) + 72 * len(sizes),
                "flops": sum(_grid_work(s, case["loads"], 200, nq) for s in sizes)}
    if do == "gradient":
        return {"bytes": 16 * N + 16 * ns * ns, "flops": _grid_work(n, 2 * ns, 250, nq)}
    if do == "finite":
        return {"bytes": 8 * N * (1 + nq * D * D), "flops": _grid_work(n, 1, 400, nq)}
    return {"bytes": 8 * N * (1 + case["loads"] * nq * ns), "flops": _grid_work(n, case["loads"], 200, nq)}


# ------------------------------------------------------------------- exact
class _Cell:
    """A periodic cell in 64 bits: gradients of a nodal field at the evaluation
    points of every voxel, their adjoint, and the inverse of B^T B.  The unit
    cell, voxel size 1/n."""

    def __init__(self, n, derivative="fe"):
        self.n, self.D, self.derivative = n, len(n), derivative
        D = self.D
        self.axes = tuple(range(-D, 0))
        if D == 2:
            self.elements = [[((1, 0), (0, 0)), ((0, 1), (0, 0))], [((1, 1), (0, 1)), ((1, 1), (1, 0))]]
        else:
            self.elements = []
            for a, b, c in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
                at = [[0, 0, 0]]
                for ax in (a, b, c):
                    at.append([v + (1 if i == ax else 0) for i, v in enumerate(at[-1])])
                e = [None] * 3
                for k, ax in enumerate((a, b, c)):
                    e[ax] = (tuple(at[k + 1]), tuple(at[k]))
                self.elements.append(e)
        self.ix = list(range(D))
        self.g = self._symbols()
        norm = sum((abs(ga) ** 2).sum(0) for ga in self.g)
        dead = norm < 1e-20 * norm.max()
        self.M = torch.zeros(D, D, *norm.shape, dtype=torch.complex128, device=DEV)
        for ga in self.g:
            self.M += 0.5 * ga[:, None] * ga[None, :].conj()
            for i in range(D):
                self.M[i, i] += 0.5 * (abs(ga) ** 2).sum(0)
        # B^H B of small strain: M_ij = 1/2 sum_t (|g|^2 delta_ij + g_i conj(g_j)), with the test index first
        self.M = self.M.conj().transpose(0, 1).contiguous()
        for i in range(D):
            self.M[i, i] = torch.where(dead, 1.0 + 0j, self.M[i, i])
        self.scalar = torch.where(dead, 1.0, norm)
        self.alive = (~dead).to(torch.float64)
        self.inv = _inverse(self.M)
        del self.M

    def _theta(self):
        out = []
        for ax in range(self.D):
            size = self.n[ax]
            k = (torch.fft.rfftfreq if ax == 0 else torch.fft.fftfreq)(size, device=DEV, dtype=torch.float64) * size
            k = k.abs() if ax == 0 else k
            out.append(k.reshape([-1 if a == self.D - 1 - ax else 1 for a in range(self.D)]))
        return out

    def _symbols(self):
        """Fourier symbols g[t][axis] of the derivative at evaluation point t."""
        k = self._theta()
        half = tuple(reversed(self.n[1:])) + (self.n[0] // 2 + 1,)
        ph = [torch.exp(2j * math.pi * k[a] / self.n[a]) for a in range(self.D)]
        if self.derivative == "fe":
            def at(c):
                v = torch.ones(half, dtype=torch.complex128, device=DEV)
                for a in range(self.D):
                    if c[a]:
                        v = v * ph[a]
                return v
            return [torch.stack([(at(p) - at(m)) * self.n[a] for a, (p, m) in enumerate(e)]) for e in self.elements]
        g = []
        for a in range(self.D):
            if self.derivative == "fourier":
                v = 2j * math.pi * torch.where(2 * k[a].abs() == self.n[a], 0.0, k[a])
            else:
                v = (ph[a] - 1) * self.n[a]
                if self.derivative == "lsq":  # the other axes averaged over the voxel's two nodes
                    for b in range(self.D):
                        if b != a:
                            v = v * (ph[b] + 1) / 2
            g.append(v.expand(half).clone())
        return [torch.stack(g)]

    def fft(self, u):
        return torch.fft.rfftn(u, dim=self.axes)

    def ifft(self, u):
        return torch.fft.irfftn(u, s=_shape(self.n), dim=self.axes)

    def _roll(self, u, c, sign):
        for a in range(self.D):
            if c[a]:
                u = torch.roll(u, sign, dims=-1 - a)
        return u

    def grad(self, u):
        """H[t][i, a] = d u_i / d x_a of u [D, *shape]."""
        if self.derivative != "fe":
            uh = self.fft(u)
            return torch.stack([torch.stack([self.ifft(uh * g[a]) for a in range(self.D)], 1) for g in self.g])
        at = {}
        out = torch.empty(len(self.elements), self.D, self.D, *u.shape[1:], dtype=u.dtype, device=u.device)
        for t, e in enumerate(self.elements):
            for a, (p, m) in enumerate(e):
                for c in (p, m):
                    if c not in at:
                        at[c] = self._roll(u, c, -1)
                out[t][:, a] = (at[p] - at[m]) * self.n[a]
        return out

    def div(self, P):
        """The adjoint of grad."""
        if self.derivative != "fe":
            return self.ifft(sum(self.fft(P[t][:, a]) * g[a].conj() for t, g in enumerate(self.g) for a in range(self.D)))
        at = {}
        for t, e in enumerate(self.elements):
            for a, (p, m) in enumerate(e):
                v = P[t][:, a] * self.n[a]
                at[p] = at[p] + v if p in at else v
                at[m] = at[m] - v if m in at else -v
        return sum(self._roll(v, c, 1) for c, v in at.items())

    def precondition(self, f, small=True):
        fh = self.fft(f) * self.alive
        if not small:
            return self.ifft(fh / self.scalar)
        return self.ifft(torch.stack([sum(self.inv[i, j] * fh[j] for j in range(self.D)) for i in range(self.D)]))

    def cg(self, apply, f, small=True, tol=2e-14, most=6000):
        """Solve apply(u) = f by preconditioned CG."""
        u, r = torch.zeros_like(f), f.clone()
        z = self.precondition(r, small)
        p, rz = z.clone(), (r * z).sum()
        first, best, since = rz.clone(), float("inf"), 0
        for it in range(most):
            q = apply(p)
            alpha = rz / (p * q).sum()
            u += alpha * p
            r -= alpha * q
            z = self.precondition(r, small)
            new = (r * z).sum()
            p = z + (new / rz) * p
            rz = new
            if it % 8 == 7:
                now = float((rz / first).clamp(min=0)) ** 0.5
                since = 0 if now < 0.5 * best else since + 1
                best = min(best, now)
                if now < tol or since > 12:
                    break
        return u


def _inverse(M):
    """Inverse of the 2 x 2 or 3 x 3 matrices M[i, j, ...] by cofactors."""
    D = M.shape[0]
    if D == 2:
        det = M[0, 0] * M[1, 1] - M[0, 1] * M[1, 0]
        rows = [[M[1, 1], -M[0, 1]], [-M[1, 0], M[0, 0]]]
    else:
        def cof(i, j):
            a, b = [k for k in range(3) if k != i]
            c, d = [k for k in range(3) if k != j]
            return (1 if (i + j) % 2 == 0 else -1) * (M[a, c] * M[b, d] - M[a, d] * M[b, c])
        rows = [[cof(j, i) for j in range(3)] for i in range(3)]
        det = sum(M[0, j] * rows[j][0] for j in range(3))
    return torch.stack([torch.stack([v / det for v in row]) for row in rows])


LAM, MU2 = NU / ((1 + NU) * (1 - 2 * NU)), 1 / (1 + NU)


def _sym(H):
    return 0.5 * (H + H.transpose(1, 2))


def _stress(E, eps):
    """Isotropic law, per evaluation point: eps [t, i, j, *shape]."""
    tr = sum(eps[:, i, i] for i in range(eps.shape[1]))
    s = MU2 * eps
    for i in range(eps.shape[1]):
        s[:, i, i] += LAM * tr
    return E * s


def _pairs(D):
    return [(0, 0), (1, 1), (0, 1)] if D == 2 else [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]


def _to_mandel(t):
    """[t, i, j, *shape] -> [t * n_s + s, N]"""
    D = t.shape[1]
    rows = [t[q, i, j] * (1.0 if i == j else math.sqrt(2.0)) for q in range(t.shape[0]) for i, j in _pairs(D)]
    return torch.stack(rows).reshape(len(rows), -1)


def _from_mandel(v, D, lead=()):
    """Symmetric tensor [..lead, D, D, *rest] of Mandel components v[..lead][n_s, *rest]."""
    out = [[None] * D for _ in range(D)]
    for s, (i, j) in enumerate(_pairs(D)):
        out[i][j] = out[j][i] = v[s] * (1.0 if i == j else 1 / math.sqrt(2.0))
    return torch.stack([torch.stack(row) for row in out])


def _solve_exact(cell, E, load):
    """Total strain [t, i, j, *shape] of one macroscopic Mandel strain."""
    D = cell.D
    em = _from_mandel(torch.as_tensor(load, dtype=torch.float64, device=DEV), D)
    em = em.reshape(1, D, D, *([1] * D))
    nq = len(cell.g)
    start = _stress(E, em.expand(nq, D, D, *_shape(cell.n)).clone())
    u = cell.cg(lambda p: cell.div(_stress(E, _sym(cell.grad(p)))), -cell.div(start))
    return em + _sym(cell.grad(u))


def _mean(t):
    """Mean over evaluation points and voxels, in Mandel components."""
    return _to_mandel(t).reshape(t.shape[0], -1, math.prod(t.shape[3:])).mean(dim=(0, 2))


def _finite_exact(cell, E):
    """Deformation gradient [t, i, a, *shape] by Newton's method."""
    D = cell.D
    Fm = torch.tensor(F_MACRO, dtype=torch.float64, device=DEV).reshape(1, D, D, *([1] * D))
    one = torch.eye(D, dtype=torch.float64, device=DEV).reshape(1, D, D, *([1] * D))

    def mul(a, b):
        return torch.einsum("tij...,tjk...->tik...", a, b)

    def second(F):
        return _stress(E, 0.5 * (mul(F.transpose(1, 2), F) - one))

    u = torch.zeros(D, *_shape(cell.n), dtype=torch.float64, device=DEV)
    first, last = None, float("inf")
    for _ in range(30):
        F = Fm + cell.grad(u)
        S = second(F)
        f = cell.div(mul(F, S))
        size = float(f.norm())
        first = size if first is None else first
        if size <= 1e-13 * first or size > 0.5 * last and size < 1e-9 * first:
            break
        last = size

        def tangent(p):
            dF = cell.grad(p)
            dE = _sym(mul(F.transpose(1, 2), dF))
            return cell.div(mul(dF, S) + mul(F, _stress(E, dE)))

        u = u + cell.cg(tangent, -f, small=False, tol=1e-9)
    F = Fm + cell.grad(u)
    return F, mul(F, second(F))


def exact(case, seed):
    n, do = _grid(case), case["do"]
    D, N = len(n), math.prod(n)
    ns = 3 if D == 2 else 6
    if do in ("solve", "gradient") and N * max(1, case["loads"]) > 4194304:
        return None  # over 20 s
    x = _inputs(case, seed)
    if do == "batch":
        out = []
        for size, E in zip(x["sizes"], x["E"]):
            cell, E = _Cell(size), torch.as_tensor(E, device=DEV)
            out.append(torch.stack([_mean(_stress(E, _solve_exact(cell, E, v))) for v in np.eye(3)], 1))
        return torch.stack(out).cpu().numpy()
    cell, E = _Cell(n, case.get("derivative", "fe")), x["E"]
    nq = len(cell.g)
    if do in ("operator", "static_op"):
        p = x["p"].to(torch.float64).reshape(nq, ns, *_shape(n)).transpose(0, 1)
        eps = _from_mandel(p, D).transpose(1, 2).transpose(0, 1)
        return _to_mandel(_sym(cell.grad(cell.precondition(cell.div(_stress(E, eps))))))
    if do == "finite":
        F, P = _finite_exact(cell, E)
        return {"P": P.mean(dim=(0, 3, 4)).reshape(1, D, D).cpu().numpy(),
                "F": F.reshape(nq, D, D, N).cpu().numpy()}
    if do == "gradient":
        eps = [_solve_exact(cell, E, v) for v in np.eye(ns)]
        C = torch.stack([_mean(_stress(E, e)) for e in eps], 1)
        grad = torch.zeros_like(E)
        for a in range(ns):  # the operator is its own adjoint: the adjoint states are the solutions themselves
            w = sum(x["W"][a, l] * eps[l] for l in range(ns))
            grad += (eps[a] * _stress(torch.ones_like(E), w)).sum(dim=(0, 1, 2))
        return {"C": C, "grad": grad / (N * nq)}
    eps = [_solve_exact(cell, E, v) for v in _loads(case)]
    return {"S": torch.stack([_mean(_stress(E, e)) for e in eps]).cpu().numpy(), "eps": [_to_mandel(e) for e in eps]}
