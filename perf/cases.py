"""Performance cases of the thermal solver: what a user's program calls, and how.

Each case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)``
one more of the same ranges, ``prepare(case, seed)`` the inputs and grid handles a
program holds before the call, ``run(state)`` one pass through the public entry
points, ``work(case)`` the bytes and operations a pass cannot do without, and
``exact(case, seed)`` the same outputs computed in FP64 by plain torch: layer-uniform
stacks by diagonalising the in-plane operator (cosine transform, one tridiagonal
system per mode), conductivity maps by conjugate gradients on the assembled faces.

Kinds:
  steady    one steady solve (plain FP64 or mixed precision)
  precond   one application of a preconditioner (Chebyshev or multigrid V-cycle)
  step      one backward-Euler step
  run       a backward-Euler trajectory whose power map switches
  batched   independent steady stacks of uneven size in one call
  adjoint   steady solve, hotspot objective and its gradient through autograd
"""
import math

import torch

from paper_2606_17850_gb300 import HotspotLSE, SteadyAdjoint, ThermalGrid, solve_batched

UM = 1e-6
DX = 50 * UM
H_TOP, T_AMB, DT = 1e4, 45.0, 1e-4
SI, BOND, TIM, CU = (150.0, 1.63e6), (2.5, 1.5e6), (4.0, 2.0e6), (400.0, 3.45e6)
T3 = 1000.0 / 3.0
# (conductivity W/mK, heat capacity J/m^3K), thickness in um, powered; bottom to top
STACKS = {
    4: ((SI, 100, True), (BOND, 10, False), (TIM, 25, False), (CU, 1000, False)),
    6: ((SI, 100, True), (BOND, 10, False), (TIM, 25, False), (CU, T3, False), (CU, T3, False), (CU, T3, False)),
    8: ((SI, 100, True), (BOND, 10, False), (SI, 100, True), (BOND, 10, False), (TIM, 25, False), (CU, T3, False),
        (CU, T3, False), (CU, T3, False)),
    10: ((SI, 10, False), (SI, 2, True), (BOND, 10, False), (BOND, 2, False), (BOND, 10, False), (SI, 2, True),
         (SI, 200, False), (TIM, 100, False), (CU, 400, False), (CU, 1000, False)),
}
CLASSES = ((128, 4), (256, 6), (384, 8), (512, 8))  # batch size classes: side, layers
# Chebyshev interval of the Jacobi-scaled transient operator at DT on these stacks
LAM_MIN, LAM_MAX = 0.05, 2.05


def listed():
    return [
        {"name": "steady-fp64-64x64x4", "kind": "steady", "nx": 64, "ny": 64, "layers": 4, "precision": "fp64",
         "precond": "cheb", "degree": 30, "graph": 1},
        {"name": "steady-mixed-64x64x4", "kind": "steady", "nx": 64, "ny": 64, "layers": 4, "precision": "mixed",
         "precond": "cheb", "degree": 30, "graph": 1},
        {"name": "steady-mg-512x512x8", "kind": "steady", "nx": 512, "ny": 512, "layers": 8, "precision": "mixed",
         "precond": "mg", "degree": 30, "graph": 1},
        {"name": "steady-cheb-301x203x8", "kind": "steady", "nx": 301, "ny": 203, "layers": 8, "precision": "mixed",
         "precond": "cheb", "degree": 30, "graph": 0},
        {"name": "precond-cheb-1024x1024x8", "kind": "precond", "nx": 1024, "ny": 1024, "layers": 8,
         "precond": "cheb", "degree": 29, "map": False},
        {"name": "precond-cheb-map-500x333x6", "kind": "precond", "nx": 500, "ny": 333, "layers": 6,
         "precond": "cheb", "degree": 16, "map": True},
        {"name": "precond-mg-640x384x8", "kind": "precond", "nx": 640, "ny": 384, "layers": 8, "precond": "mg",
         "degree": 1, "map": False},
        {"name": "step-130x70x4", "kind": "step", "nx": 130, "ny": 70, "layers": 4, "degree": 12},
        {"name": "run-1024x1024x8", "kind": "run", "nx": 1024, "ny": 1024, "layers": 8, "degree": 29, "steps": 100,
         "steps_per_map": 25, "map": False},
        {"name": "run-map-256x256x6", "kind": "run", "nx": 256, "ny": 256, "layers": 6, "degree": 29, "steps": 40,
         "steps_per_map": 10, "map": True},
        {"name": "batched-mg-32", "kind": "batched", "count": 32, "classes": 4, "scale": 1, "precond": "mg",
         "degree": 30},
        {"name": "adjoint-mg-1024x1024x10", "kind": "adjoint", "nx": 1024, "ny": 1024, "layers": 10},
    ]


def _side(rng, lo, hi):
    """A side of the range, spread over its logarithm: multiples of 4 and odd ones alike."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return v if rng.random() < 0.4 else max(lo, v // 4 * 4)


def draw(rng):
    kind = rng.choice(["steady", "steady", "precond", "precond", "step", "run", "batched", "adjoint"])
    c = {"kind": kind}
    if kind == "batched":
        scale = rng.choice([1, 2, 4])
        return dict(c, count=rng.randint(3, 32), classes=rng.randint(1, 1 << 16), scale=scale,
                    precond="mg" if scale == 1 else rng.choice(["mg", "cheb"]), degree=rng.randint(16, 32))
    top = {"steady": 512, "precond": 1024, "step": 1024, "run": 512, "adjoint": 768}[kind]
    low = 128 if kind == "adjoint" else 48
    c.update(nx=_side(rng, low, top), ny=_side(rng, low, top), layers=rng.choice([4, 6, 8, 8]))
    if kind == "steady":
        fp64 = rng.random() < 0.25
        if fp64:
            c.update(nx=min(c["nx"], 256), ny=min(c["ny"], 256))
        c.update(precision="fp64" if fp64 else "mixed", precond="cheb" if fp64 else rng.choice(["cheb", "mg"]),
                 degree=rng.randint(10, 32), graph=rng.randint(0, 1))
    elif kind == "precond":
        pc = rng.choice(["cheb", "cheb", "mg"])
        c.update(precond=pc, degree=rng.randint(6, 32) if pc == "cheb" else 1, map=rng.random() < 0.4)
    elif kind == "step":
        c.update(degree=rng.randint(6, 24))
    elif kind == "run":
        c.update(degree=rng.randint(12, 30), steps=rng.randint(10, 60), steps_per_map=rng.randint(5, 25),
                 map=rng.random() < 0.4)
    else:
        c.update(layers=rng.choice([8, 10, 10]))
    return c


# ---------------------------------------------------------------- inputs


def _stack(layers):
    k = [m[0] for m, _, _ in STACKS[layers]]
    c = [m[1] for m, _, _ in STACKS[layers]]
    dz = [t * UM for _, t, _ in STACKS[layers]]
    return k, c, dz, [i for i, s in enumerate(STACKS[layers]) if s[2]]


def _gen(seed):
    g = torch.Generator()
    g.manual_seed(int(seed))
    return g


def _u(g, lo, hi):
    return lo + (hi - lo) * torch.rand((), generator=g).item()


def _floorplan(nx, ny, g, rects=64, spots=16):
    """Block floorplan with Gaussian hotspots, W/cm^2 (ny, nx)."""
    q = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    side = lambda n: int(_u(g, max(1, n // 32), max(1, n // 4) + 1))  # noqa: E731
    for _ in range(rects):
        w, h = min(side(nx), nx), min(side(ny), ny)
        x0, y0 = int(_u(g, 0, nx - w + 1)), int(_u(g, 0, ny - h + 1))
        q[y0:y0 + h, x0:x0 + w] = _u(g, 5.0, 80.0)
    xs = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) * DX
    ys = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) * DX
    for _ in range(spots):
        cx, cy, s, p = _u(g, 0, nx * DX), _u(g, 0, ny * DX), _u(g, 100, 300) * UM, _u(g, 200.0, 500.0)
        q += p * torch.outer(torch.exp(-((ys - cy) ** 2) / (2 * s * s)), torch.exp(-((xs - cx) ** 2) / (2 * s * s)))
    return q


def _power(nx, ny, layers, g, dtype=torch.float32):
    """Power map in W per cell, flat, x fastest."""
    p = torch.zeros(layers, ny, nx, dtype=torch.float64, device="cuda")
    for z in _stack(layers)[3]:
        p[z] = _floorplan(nx, ny, g) * 1e4 * DX * DX
    return p.reshape(-1).to(dtype)


def _kmap(nx, ny, layers, seed):
    """Per-cell conductivities: each layer's value times U[0.8, 1.2]."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) + 77)
    f = 0.8 + 0.4 * torch.rand(layers, ny, nx, generator=g, device="cuda", dtype=torch.float64)
    return (f * torch.tensor(_stack(layers)[0], dtype=torch.float64, device="cuda")[:, None, None]).reshape(-1)


def _normal(n, seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) + 5)
    return torch.randn(n, generator=g, device="cuda", dtype=dtype)


def _grid(nx, ny, layers, k=None):
    k0, c, dz, _ = _stack(layers)
    return ThermalGrid(nx, ny, k if k is not None else k0, c, H_TOP, DX, DX, dz, T_AMB)


def _instances(case):
    """(side, layers) of every stack of a batch."""
    g = _gen(case["classes"])
    return [(CLASSES[i][0] // case["scale"], CLASSES[i][1])
            for i in torch.randint(0, 4, (case["count"],), generator=g).tolist()]


def _batch_inputs(case, seed):
    """Per stack: side, layers, conductivities (each +-20 %) and power map."""
    out = []
    for i, (side, L) in enumerate(_instances(case)):
        g = _gen(1000 * seed + i)
        k = [v * _u(g, 0.8, 1.2) for v in _stack(L)[0]]
        out.append((side, L, k, _power(side, side, L, g)))
    return out


def _inputs(case, seed):
    """The tensors of a single-grid case."""
    nx, ny, L, kind = case["nx"], case["ny"], case["layers"], case["kind"]
    n = nx * ny * L
    g = _gen(seed)
    s = {}
    if case.get("map"):
        s["kmap"] = _kmap(nx, ny, L, seed)
    if kind == "precond":
        s["r"] = _normal(n, seed, torch.float32)
    elif kind == "run":
        s["maps"] = [_power(nx, ny, L, g) for _ in range(4)]
        s["T0"] = torch.full((n,), T_AMB, dtype=torch.float64, device="cuda")
    else:
        s["power"] = _power(nx, ny, L, g)
        if kind == "step":  # a warm state with the power map's pattern
            rise = s["power"].double().reshape(L, ny, nx).sum(0) * 2e3
            s["T"] = (T_AMB + 2.0 + rise).expand(L, ny, nx).reshape(-1).contiguous()
        if kind == "adjoint":
            s["k"] = [v * _u(g, 0.9, 1.1) for v in _stack(L)[0]]
    return s


def _opts(case):
    kind = case["kind"]
    if kind == "steady":
        return dict(precision=case["precision"], precond=case["precond"], cheb_degree=case["degree"],
                    use_graph=case["graph"], tol_rel=1e-10 if case["precision"] == "fp64" else 1e-8)
    if kind == "precond":
        o = dict(precond=case["precond"], cheb_degree=case["degree"])
        if case["precond"] == "cheb":
            o.update(cheb_lam_min=LAM_MIN, cheb_lam_max=LAM_MAX)
        return o
    if kind == "step":
        return dict(cheb_degree=case["degree"], tol_rel=1e-8)
    if kind == "run":
        return dict(cheb_degree=case["degree"], guess=3, use_graph=1, tol_rel=1e-8)
    if kind == "batched":
        return dict(precond=case["precond"], cheb_degree=case["degree"], tol_rel=1e-8)
    return dict(precond="mg", use_graph=1, tol_rel=1e-9)


def prepare(case, seed):
    s = {"kind": case["kind"], "opts": _opts(case)}
    if case["kind"] == "batched":
        inst = _batch_inputs(case, seed)
        s["grids"] = [_grid(side, side, L, k) for side, L, k, _ in inst]
        s["powers"] = [p for _, _, _, p in inst]
        s["Ts"] = [torch.empty(g.n, dtype=torch.float64, device="cuda") for g in s["grids"]]
        return s
    s.update(_inputs(case, seed))
    s["grid"] = _grid(case["nx"], case["ny"], case["layers"])
    if "kmap" in s:
        s["grid"].set_conductivity_map(s["kmap"])
    if case["kind"] == "precond":
        s["dt"] = DT if case["precond"] == "cheb" else 0.0
    elif case["kind"] == "run":
        s["steps"], s["steps_per_map"] = case["steps"], case["steps_per_map"]
    elif case["kind"] == "adjoint":
        s["layers"] = _stack(case["layers"])[3]
        s["power"].requires_grad_(True)
        s["k"] = torch.tensor(s["k"], dtype=torch.float64, requires_grad=True)
    return s


def run(s):
    kind, o = s["kind"], s["opts"]
    if kind == "steady":
        return s["grid"].solve_steady(s["power"], **o)[0]
    if kind == "precond":
        return s["grid"].precond(s["r"], s["dt"], **o)
    if kind == "step":
        return s["grid"].step_transient(s["power"], DT, s["T"].clone(), **o)[0]
    if kind == "run":
        return s["grid"].run_transient(s["maps"], s["steps_per_map"], s["steps"], DT, s["T0"].clone(), **o)[0]
    if kind == "batched":
        solve_batched(s["grids"], s["powers"], s["Ts"], **o)
        return s["Ts"]
    T = SteadyAdjoint.apply(s["grid"], s["power"], s["k"], o)
    J = HotspotLSE.apply(s["grid"], T, s["layers"], 2.0)
    dP, dk = torch.autograd.grad(J, (s["power"], s["k"]))
    return {"T": T.detach(), "J": J.detach(), "dJdP": dP, "dJdk": dk}


def work(case):
    """Inputs read once, outputs written once; the operations of one preconditioner
    application and one product per system (an iterative solve needs at least that)."""
    kind = case["kind"]
    if kind == "batched":
        n = sum(a * a * L for a, L in _instances(case))
        pc, bytes_ = 80 if case["precond"] == "mg" else 11 * (case["degree"] - 1), 12 * n
    else:
        n = case["nx"] * case["ny"] * case["layers"]
        mg = case.get("precond") == "mg" or kind == "adjoint"
        pc = 80 if mg else 11 * (case["degree"] - 1)
        bytes_ = {"steady": 12 * n, "precond": 8 * n, "step": 20 * n, "adjoint": 32 * n}.get(kind, 0)
        if kind == "run":
            maps = min(4, -(-case["steps"] // case["steps_per_map"]))
            bytes_ = (4 * maps + 16) * n
        if case.get("map"):
            bytes_ += 12 * n  # the face conductances
    if kind == "precond":
        return {"bytes": bytes_, "flops": pc * n}
    systems = {"run": case.get("steps", 1), "adjoint": 2}.get(kind, 1)
    return {"bytes": bytes_, "flops": systems * (pc + 13) * n}


# ---------------------------------------------------------------- FP64 reference (plain torch)


def _layer_faces(k, dz):
    """gx (= gy) per layer and gz between layers z and z + 1, square cells of side DX."""
    k, dz = torch.tensor(k, dtype=torch.float64, device="cuda"), torch.tensor(dz, dtype=torch.float64, device="cuda")
    S = DX * DX
    return k * dz, S / (dz[:-1] / (2 * k[:-1]) + dz[1:] / (2 * k[1:]))


def _layer_diag(c, dz, dt):
    s = torch.zeros(len(dz), dtype=torch.float64, device="cuda")
    s[-1] = H_TOP * DX * DX
    cap = torch.zeros_like(s)
    if dt > 0:
        cap = torch.tensor(c, dtype=torch.float64, device="cuda") * torch.tensor(
            dz, dtype=torch.float64, device="cuda") * (DX * DX / dt)
    return s + cap, cap


class _Modes:
    """(A theta = b) on a layer-uniform grid: cosine modes in x and y, Thomas in z."""

    def __init__(self, nx, ny, k, c, dz, dt=0.0):
        self.C = [self._dct(ny), self._dct(nx)]
        ax, ay = self._eig(nx), self._eig(ny)
        g, gz = _layer_faces(k, dz)
        s, self.cap = _layer_diag(c, dz, dt)
        L = len(dz)
        self.gz, self.L = gz, L
        w, self.m, wprev = [], [], None
        for z in range(L):
            b = s[z] + g[z] * (ax[None, :] + ay[:, None])
            if z + 1 < L:
                b = b + gz[z]
            if z > 0:
                b = b + gz[z - 1] - gz[z - 1] * wprev
            self.m.append(1.0 / b)
            wprev = gz[z] * self.m[z] if z + 1 < L else None
            w.append(wprev)
        self.w = w

    @staticmethod
    def _eig(n):
        return 2 - 2 * torch.cos(math.pi * torch.arange(n, dtype=torch.float64, device="cuda") / n)

    @staticmethod
    def _dct(n):
        i = torch.arange(n, dtype=torch.float64, device="cuda")
        c = torch.cos(math.pi * i[:, None] * (i[None, :] + 0.5) / n) * math.sqrt(2.0 / n)
        c[0] /= math.sqrt(2.0)
        return c

    def to(self, f):
        return self.C[0] @ f @ self.C[1].T

    def back(self, f):
        return self.C[0].T @ f @ self.C[1]

    def solve(self, b):
        """Tridiagonal solves of every mode: b (L, ny, nx) in mode space."""
        d = []
        for z in range(self.L):
            t = b[z] if z == 0 else b[z] + self.gz[z - 1] * d[z - 1]
            d.append(t * self.m[z])
        for z in range(self.L - 2, -1, -1):
            d[z] = d[z] + self.w[z] * d[z + 1]
        return torch.stack(d)


class _Faces:
    """The operator from per-face arrays (L, ny, nx): faces towards +x, +y, +z."""

    def __init__(self, gx, gy, gz, s):
        self.gx, self.gy, self.gz, self.s = gx, gy, gz, s
        d = s.clone()
        for g, dim in ((gx, 2), (gy, 1), (gz, 0)):
            n = d.shape[dim]
            d += g
            d.narrow(dim, 1, n - 1).add_(g.narrow(dim, 0, n - 1))
        self.diag = d

    @classmethod
    def of_case(cls, case, dt, kmap=None):
        nx, ny, L = case["nx"], case["ny"], case["layers"]
        k0, c, dz, _ = _stack(L)
        k = kmap.reshape(L, ny, nx) if kmap is not None else torch.tensor(
            k0, dtype=torch.float64, device="cuda")[:, None, None].expand(L, ny, nx)
        t = torch.tensor(dz, dtype=torch.float64, device="cuda")[:, None, None]
        gx, gy, gz = (torch.zeros(L, ny, nx, dtype=torch.float64, device="cuda") for _ in range(3))
        gx[:, :, :-1] = DX * t / (DX / (2 * k[:, :, :-1]) + DX / (2 * k[:, :, 1:]))
        gy[:, :-1] = DX * t / (DX / (2 * k[:, :-1]) + DX / (2 * k[:, 1:]))
        gz[:-1] = DX * DX / (t[:-1] / (2 * k[:-1]) + t[1:] / (2 * k[1:]))
        s, cap = _layer_diag(c, dz, dt)
        f = cls(gx, gy, gz, s[:, None, None].expand(L, ny, nx).clone())
        f.cap = cap[:, None, None]
        return f

    def apply(self, v):
        y = self.s * v
        for g, dim in ((self.gx, 2), (self.gy, 1), (self.gz, 0)):
            n = v.shape[dim]
            if n < 2:
                continue
            a, b = v.narrow(dim, 0, n - 1), v.narrow(dim, 1, n - 1)
            f = g.narrow(dim, 0, n - 1) * (a - b)
            y.narrow(dim, 0, n - 1).add_(f)
            y.narrow(dim, 1, n - 1).sub_(f)
        return y

    def solve(self, b, x, tol=1e-13, most=4000):
        """Jacobi-preconditioned conjugate gradients from the guess x."""
        r = b - self.apply(x)
        stop = tol * b.norm().item()
        z = r / self.diag
        p, rz = z, (r * z).sum()
        for it in range(most):
            q = self.apply(p)
            a = rz / (p * q).sum()
            x = x + a * p
            r = r - a * q
            if it % 10 == 9 and r.norm().item() <= stop:
                break
            z = r / self.diag
            rz, old = (r * z).sum(), rz
            p = z + (rz / old) * p
        return x

    def thomas(self, b):
        """T^-1 b, T the tridiagonal block of every column."""
        d, w, L = [], [], b.shape[0]
        for z in range(L):
            piv, t = self.diag[z], b[z]
            if z > 0:
                piv, t = piv - self.gz[z - 1] * w[z - 1], t + self.gz[z - 1] * d[z - 1]
            w.append(self.gz[z] / piv)
            d.append(t / piv)
        for z in range(L - 2, -1, -1):
            d[z] = d[z] + w[z] * d[z + 1]
        return torch.stack(d)

    def coarse(self):
        """Galerkin operator of 2 x 2-column aggregates."""
        L, ny, nx = self.s.shape
        py, px = ny % 2, nx % 2
        pad = lambda t: torch.nn.functional.pad(t, (0, px, 0, py))  # noqa: E731
        four = lambda t: _pool(pad(t))  # noqa: E731
        gx, gy = pad(self.gx)[:, :, 1::2], pad(self.gy)[:, 1::2, :]
        gx = gx[:, 0::2] + gx[:, 1::2]
        gy = gy[:, :, 0::2] + gy[:, :, 1::2]
        return _Faces(gx, gy, four(self.gz), four(self.s))

    def vcycle(self, b, omega=0.8):
        L, ny, nx = b.shape
        if max(nx, ny) <= 8:
            n = L * ny * nx
            eye = torch.eye(n, dtype=torch.float64, device="cuda").reshape(n, L, ny, nx)
            A = torch.stack([self.apply(e).reshape(-1) for e in eye])
            return torch.linalg.solve(A, b.reshape(-1)).reshape(b.shape)
        x = omega * self.thomas(b)
        r = torch.nn.functional.pad(b - self.apply(x), (0, nx % 2, 0, ny % 2))
        e = self.coarse().vcycle(_pool(r), omega)
        x = x + e.repeat_interleave(2, 1).repeat_interleave(2, 2)[:, :ny, :nx]
        return x + omega * self.thomas(b - self.apply(x))


def _pool(t):
    return t[:, 0::2, 0::2] + t[:, 0::2, 1::2] + t[:, 1::2, 0::2] + t[:, 1::2, 1::2]


def _chebyshev(A, r, degree):
    """Degree-`degree` Chebyshev polynomial of D^-1 A on [LAM_MIN, LAM_MAX] applied to r."""
    theta, delta = 0.5 * (LAM_MAX + LAM_MIN), 0.5 * (LAM_MAX - LAM_MIN)
    sigma = theta / delta
    rho, zp, z = 1 / sigma, torch.zeros_like(r), r / A.diag / theta
    for _ in range(1, degree):
        new = 1 / (2 * sigma - rho)
        z, zp = z + new * rho * (z - zp) + (2 * new / delta) * ((r - A.apply(z)) / A.diag), z
        rho = new
    return z


def exact(case, seed):
    if case["kind"] == "batched":
        out = []
        for side, L, k, p in _batch_inputs(case, seed):
            _, c, dz, _ = _stack(L)
            m = _Modes(side, side, k, c, dz)
            out.append(T_AMB + m.back(m.solve(m.to(p.double().reshape(L, side, side)))).reshape(-1))
        return out
    nx, ny, L, kind = case["nx"], case["ny"], case["layers"], case["kind"]
    k, c, dz, powered = _stack(L)
    s = _inputs(case, seed)
    cells = lambda t: t.double().reshape(L, ny, nx)  # noqa: E731
    if kind == "precond":
        A = _Faces.of_case(case, DT if case["precond"] == "cheb" else 0.0, s.get("kmap"))
        r = cells(s["r"])
        return (_chebyshev(A, r, case["degree"]) if case["precond"] == "cheb" else A.vcycle(r)).reshape(-1)
    if kind == "steady":
        m = _Modes(nx, ny, k, c, dz)
        return T_AMB + m.back(m.solve(m.to(cells(s["power"])))).reshape(-1)
    if kind == "step":
        m = _Modes(nx, ny, k, c, dz, DT)
        b = cells(s["power"]) + m.cap[:, None, None] * (cells(s["T"]) - T_AMB)
        return T_AMB + m.back(m.solve(m.to(b))).reshape(-1)
    if kind == "run":
        at = lambda i: (i // case["steps_per_map"]) % 4  # noqa: E731
        if case["map"]:
            A = _Faces.of_case(case, DT, s["kmap"])
            th = torch.zeros(L, ny, nx, dtype=torch.float64, device="cuda")
            for i in range(case["steps"]):
                th = A.solve(cells(s["maps"][at(i)]) + A.cap * th, th)
            return T_AMB + th.reshape(-1)
        m = _Modes(nx, ny, k, c, dz, DT)
        maps = [m.to(cells(p)) for p in s["maps"]]
        th = torch.zeros(L, ny, nx, dtype=torch.float64, device="cuda")
        for i in range(case["steps"]):
            th = m.solve(maps[at(i)] + m.cap[:, None, None] * th)
        return T_AMB + m.back(th).reshape(-1)
    # adjoint: J = log sum exp(2 T) / 2 over the powered layers, lambda = G^-1 dJ/dT
    k = s["k"]
    m = _Modes(nx, ny, k, c, dz)
    T = T_AMB + m.back(m.solve(m.to(cells(s["power"]))))
    hot = T[powered]
    J = torch.logsumexp(2.0 * hot.reshape(-1), 0) / 2.0
    g = torch.zeros_like(T)
    g[powered] = torch.exp(2.0 * (hot - J))
    lam = m.back(m.solve(m.to(g)))
    kt = torch.tensor(k, dtype=torch.float64, device="cuda")
    tz = torch.tensor(dz, dtype=torch.float64, device="cuda")
    gxy, gz = _layer_faces(k, dz)
    inplane = ((lam[:, :, 1:] - lam[:, :, :-1]) * (T[:, :, 1:] - T[:, :, :-1])).sum((1, 2)) + (
        (lam[:, 1:] - lam[:, :-1]) * (T[:, 1:] - T[:, :-1])).sum((1, 2))
    vert = ((lam[1:] - lam[:-1]) * (T[1:] - T[:-1])).sum((1, 2))
    dk = gxy / kt * inplane
    S = DX * DX
    dk[:-1] += vert * gz * gz / S * tz[:-1] / (2 * kt[:-1] ** 2)
    dk[1:] += vert * gz * gz / S * tz[1:] / (2 * kt[1:] ** 2)
    return {"T": T.reshape(-1), "J": J, "dJdP": lam.reshape(-1), "dJdk": (-dk).cpu()}
