"""The work that users of this package have it do, as cases to be timed.

A case is a short run: the state is initialised from FP64 device arrays,
advanced a few two-stage steps and read back (``State.init``, ``step``,
``get``), the same through host buffers (``step_host``), or one adjoint step
(``adjoint_step``).  The problems are those of the package's tests and
benchmark: density waves, shock tubes, batches of uneven cubes, the viscous
sphere, the isentropic vortex, walled channels.

``exact`` restates the method in plain FP64 torch operations (geometry,
stencils, reconstruction, kinetic flux, two-stage update), with autograd for
the adjoint; it uses none of the package's solver code.
"""
import functools
import math

import numpy as np
import torch

from paper_2102_01366_gb300 import gks
from paper_2102_01366_gb300 import inputs as I

GAMMA = 1.4
K_INT = (5.0 - 3.0 * GAMMA) / (GAMMA - 1.0)
OPEN, SLIP, FIXED, NOSLIP = I.BC_OPEN, I.BC_SLIP_WALL, I.BC_FIXED, I.BC_NOSLIP_WALL


def _case(problem, nx, ny, nz, call="step", steps=1, precision=1, weno=1, order=3, viscous=0, constraint=0,
          members=1, name=None):
    c = dict(problem=problem, nx=nx, ny=ny, nz=nz, call=call, steps=steps, precision=precision, weno=weno,
             order=order, viscous=viscous, constraint=constraint, members=members)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a shock tube small enough that a step is a row of short launches
        # (parameter sweeps, the small runs of the test suite): FP32 bulk
        _case("tube", 16, 4, 4, steps=8, name="tube_fp32_1536"),
        # the accuracy study's smallest mesh: FP64, linear weights, ten steps
        _case("wave", 8, 8, 8, steps=10, precision=0, weno=0, name="wave_fp64_3072"),
        # second-order reconstruction between slip walls, an uneven mesh
        _case("channel_slip", 37, 5, 3, steps=4, order=2, name="slip_fp32_o2_3330"),
        # the shock tube of the benchmark, FP32 bulk: the ordinary call
        _case("tube", 64, 8, 8, steps=2, name="tube_fp32_24576"),
        # the same run in FP64, the precision that results are checked in
        _case("tube", 64, 8, 8, steps=1, precision=0, name="tube_fp64_24576"),
        # a caller with host arrays: copies in, one FP64 step, copies out
        _case("tube", 45, 7, 5, call="host", precision=0, name="host_fp64_9450"),
        # independent cubes of uneven size advanced in one batch, FP32 bulk
        _case("batch", 8, 22, 0, steps=2, members=12, name="batch_fp32_12"),
        # a batch with the stencil operators kept in FP64
        _case("batch", 7, 17, 0, precision=2, members=5, name="batch_ops64_5"),
        # viscous flow past a sphere: constrained non-slip walls, far field,
        # Prandtl fix
        _case("sphere", 31, 40, 80, steps=1, viscous=1, constraint=1, name="sphere_fp32_580k"),
        # the vortex at its full size, the FP32 primal of a gradient run
        _case("vortex", 64, 64, 64, steps=1, weno=0, name="vortex_fp32_1573k"),
        # one reverse step of a gradient run (linear weights, inviscid)
        _case("vortex", 20, 20, 20, call="adjoint", precision=0, weno=0, name="adjoint_vortex_48k"),
        # reverse step with nonlinear weights, viscosity and non-slip walls
        _case("channel_noslip", 29, 9, 7, call="adjoint", precision=0, viscous=1, name="adjoint_walls_11k"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "tube", "wave", "slip", "batch", "sphere", "vortex", "host", "adjoint", "adjoint"])
    if kind == "tube":
        p = rng.choice([0, 1, 1, 2])
        ny = _log(rng, 4, 10 if p else 7)
        return _case("tube", _log(rng, 14, 150 if p == 1 else 60), ny, _log(rng, 4, 10 if p else 7),
                     steps=rng.randint(1, 2), precision=p)
    if kind == "wave":
        p = rng.choice([0, 1])
        hi = 44 if p else 14
        return _case("wave", _log(rng, 5, hi), _log(rng, 5, hi), _log(rng, 5, hi), steps=rng.randint(1, 3),
                     precision=p, weno=rng.randint(0, 1))
    if kind == "slip":
        return _case("channel_slip", _log(rng, 9, 70), _log(rng, 3, 9), _log(rng, 3, 9), steps=rng.randint(1, 3),
                     precision=rng.choice([0, 1]), order=rng.choice([2, 3]))
    if kind == "batch":
        lo = rng.randint(4, 9)
        return _case("batch", lo, lo + rng.randint(3, 14), rng.randint(0, 1000), steps=rng.randint(1, 2),
                     precision=rng.choice([1, 1, 2]), members=rng.randint(2, 13))
    if kind == "sphere":
        return _case("sphere", rng.randint(9, 30), 2 * rng.randint(7, 20), 4 * rng.randint(6, 19), viscous=1,
                     constraint=rng.randint(0, 1))
    if kind == "vortex":
        p = rng.choice([0, 1])
        n = 52 if p else 26
        return _case("vortex", _log(rng, 10, n), _log(rng, 10, n), _log(rng, 10, n), precision=p, weno=0)
    if kind == "host":
        return _case("tube", _log(rng, 14, 70), _log(rng, 4, 8), _log(rng, 4, 8), call="host", precision=0)
    if rng.random() < 0.5:
        return _case("vortex", _log(rng, 6, 21), _log(rng, 6, 21), _log(rng, 6, 21), call="adjoint", precision=0,
                     weno=rng.randint(0, 1))
    return _case("channel_noslip", _log(rng, 8, 40), _log(rng, 4, 9), _log(rng, 4, 9), call="adjoint", precision=0,
                 weno=rng.randint(0, 1), viscous=1)


# ------------------------------------------------------------- problems --

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


@functools.lru_cache(maxsize=1)
def _mesh(problem, nx, ny, nz, members):
    """Vertices, connectivity and boundary kinds; a program makes them once
    for all of its runs."""
    if problem == "sphere":
        # layers that grow by 8 % each from the wall to the far field
        return I.sphere_shell_mesh(nx, ny, nz, 0.5, 20.0, 1.08)
    if problem == "batch":
        rng = np.random.Generator(np.random.PCG64(1000 * nx + 10 * ny + nz))
        ns = rng.integers(nx, ny + 1, size=members)
        return I.batch_mesh([I.box_mesh((int(n),) * 3, seed=k, diagonal=(1, 1, -1)) for k, n in enumerate(ns)])
    if problem == "vortex":
        return I.box_mesh((nx, ny, nz), (10.0,) * 3, seed=8)
    if problem == "wave":
        return I.box_mesh((nx, ny, nz), seed=1, diagonal=(1, 1, -1))
    if problem == "tube":
        return I.box_mesh((nx, ny, nz), (1.0, 0.1, 0.1), (False, True, True), seed=2)
    m = I.box_mesh((nx, ny, nz), (1.0, ny / nx, nz / nx), (False, True, True), seed=3)
    kind = SLIP if problem == "channel_slip" else NOSLIP
    m["bkind"] = I.boundary_kinds(m, {(0, "lo"): kind, (0, "hi"): kind})
    return m


@functools.lru_cache(maxsize=1)
def _gks_mesh(problem, nx, ny, nz, members):
    return gks.Mesh(_mesh(problem, nx, ny, nz, members))


def _key(case):
    return tuple(case[k] for k in ("problem", "nx", "ny", "nz", "members"))


def _mu(case):
    if not case["viscous"]:
        return 0.0
    return 0.002


def _params(case):
    # the viscous sphere runs at the Prandtl number of air
    pr = 0.72 if case["problem"] == "sphere" else 1.0
    return gks.params(cfl=0.5, mu=_mu(case), weno=case["weno"], order=case["order"], viscous=case["viscous"],
                      precision=case["precision"], prandtl=pr, wall_constraint=case["constraint"])


def _vertices(mesh):
    dev = _device()
    tet = torch.as_tensor(mesh["tet"], device=dev)
    period = torch.as_tensor(np.asarray(mesh["period"], np.float64), device=dev)
    if period.ndim == 2:
        period = period[torch.as_tensor(mesh["case"], device=dev).long()][:, None, :]
    shift = torch.as_tensor(mesh["shift"], device=dev).double()
    return torch.as_tensor(mesh["xyz"], device=dev)[tet] + shift * period


def _prim_field(case, mesh, rng):
    """rho, u, v, w, p as functions of the position (and the cell's case)."""
    problem = case["problem"]
    r = lambda lo, hi: float(rng.uniform(lo, hi))  # noqa: E731
    if problem == "wave":
        amp, ph = r(0.1, 0.3), r(0.0, 6.28)

        def f(x):
            rho = 1.0 + amp * torch.sin(2 * math.pi * (x[..., 0] + x[..., 1] + x[..., 2]) + ph)
            one = torch.ones_like(rho)
            return rho, one, one, one, one
        return f
    if problem == "tube":
        # Sod's waves some time after the jump, smeared over about a cell as
        # the scheme carries them, over a slight transverse motion
        t, x0, ph, h = r(0.08, 0.16), r(0.45, 0.55), r(0.0, 6.28), 1.0 / case["nx"]

        def f(x):
            xi = (x[..., 0] - x0) / t
            shock = 0.5 * (1.0 + torch.tanh((xi - 1.7522) * t / h))
            contact = 0.5 * (1.0 + torch.tanh((xi - 0.9275) * t / (1.5 * h)))
            fan = torch.sigmoid((xi + 0.6267) * (6.0 / 1.113))
            rho = 1.0 + fan * (0.42632 - 1.0) + contact * (0.26557 - 0.42632) + shock * (0.125 - 0.26557)
            p = 1.0 + fan * (0.30313 - 1.0) + shock * (0.1 - 0.30313)
            u = 0.92745 * (fan - shock)
            v = 2e-3 * torch.sin(20 * math.pi * x[..., 1] + ph) * fan * (1 - shock)
            w = 2e-3 * torch.cos(20 * math.pi * x[..., 2] + ph) * fan * (1 - shock)
            return rho, u, v, w, p
        return f
    if problem == "vortex":
        s, ma, cx, cy = r(4.0, 5.0), r(0.4, 0.6), r(4.5, 5.5), r(4.5, 5.5)

        def f(x):
            dx, dy = x[..., 0] - cx, x[..., 1] - cy
            r2 = dx * dx + dy * dy
            k = s / (2 * math.pi) * torch.exp(0.5 * (1.0 - r2))
            ui = ma / math.sqrt(3.0)
            tt = 1.0 / GAMMA - (GAMMA - 1) / GAMMA * s * s / (8 * math.pi ** 2) * torch.exp(1.0 - r2)
            rho = (GAMMA * tt) ** (1.0 / (GAMMA - 1.0))
            return rho, ui - k * dy, ui + k * dx, torch.full_like(dx, ui), rho * tt
        return f
    if problem == "sphere":
        # potential flow past the sphere, retarded in a layer at the wall
        ma, d, ph = r(0.18, 0.22), r(0.15, 0.3), r(0.0, 6.28)

        def f(x):
            rr = torch.sqrt((x * x).sum(-1))
            q = 0.5 * (0.5 / rr) ** 3
            n = x / rr[..., None]
            fac = ma * (1.0 - torch.exp(-(rr - 0.47) / d))
            e = torch.tensor([1.0, 0.0, 0.0], device=x.device, dtype=x.dtype)
            vel = fac[..., None] * (e + q[..., None] * (e - 3.0 * n[..., :1] * n))
            vel = vel + 2e-3 * torch.sin(x + ph) * torch.exp(-(rr[..., None] - 0.5))
            u2 = (vel * vel).sum(-1)
            p = 1.0 / GAMMA + 0.5 * (ma * ma - u2)
            rho = (GAMMA * p) ** (1.0 / GAMMA)
            return rho, vel[..., 0], vel[..., 1], vel[..., 2], p
        return f
    if problem == "batch":
        n = int(mesh["ncase"])
        dev = _device()
        case_of = torch.as_tensor(mesh["case"], device=dev).long()
        draw1 = lambda lo, hi: torch.as_tensor(rng.uniform(lo, hi, n), device=dev)[case_of]  # noqa: E731
        slab = (torch.as_tensor(rng.permutation(n), device=dev) % 2)[case_of].double()
        mach, ph, amp = draw1(0.5, 3.0), draw1(0.0, 1.0), draw1(0.1, 0.3)
        h = torch.as_tensor(np.cbrt(6.0 / np.asarray(mesh["case_cells"])), device=dev)[case_of]

        def f(x):
            s = (x[..., 0] + ph) % 1.0
            ins = 0.5 * (torch.tanh((s - 0.25) / h) - torch.tanh((s - 0.75) / h))
            wave = 1.0 + amp * torch.sin(2 * math.pi * (x[..., 0] + x[..., 1] + x[..., 2] + ph))
            rho = slab * (0.5 + 0.5 * ins) + (1 - slab) * wave
            p = slab * (0.6 + 0.4 * ins) + (1 - slab)
            u = slab * mach * math.sqrt(GAMMA) + (1 - slab)
            return rho, u, 1 - slab, 1 - slab, p
        return f
    if problem == "channel_slip":
        # gas thrown against the walls, with a slight cross motion
        u0, ph, b, c = r(0.3, 0.8), r(0.0, 6.28), 2 * math.pi * case["nx"] / case["ny"], 2 * math.pi * case["nx"] / case["nz"]

        def f(x):
            s = torch.sin(math.pi * x[..., 0])
            rho = 1.0 + 0.1 * torch.cos(2 * math.pi * x[..., 0] + ph)
            return rho, u0 * s, 0.02 * s * torch.sin(b * x[..., 1]), 0.02 * s * torch.cos(c * x[..., 2]), 1.0 + 0.05 * s
        return f
    # decaying shear between non-slip walls
    a, ph, b = r(0.05, 0.15), r(0.0, 6.28), 2 * math.pi * case["nx"] / case["ny"]

    def f(x):
        s = torch.sin(math.pi * x[..., 0])
        rho = 1.0 + 0.02 * torch.cos(b * x[..., 1] + ph)
        return rho, 0.02 * s * torch.sin(b * x[..., 1]), a * s, 0.01 * s * s, 1.0 + 0.01 * torch.cos(math.pi * x[..., 0])
    return f


def _fields(case, seed):
    """W [5, nc] and dW [15, nc] (row 3 q + i), FP64 on the device: the
    field at the cell centroids and its central differences there."""
    mesh = _mesh(*_key(case))
    cen = _vertices(mesh).mean(1)
    prim = _prim_field(case, mesh, np.random.Generator(np.random.PCG64(seed)))

    def cons(x):
        rho, u, v, w, p = prim(x)
        return torch.stack([rho, rho * u, rho * v, rho * w, p / (GAMMA - 1) + 0.5 * rho * (u * u + v * v + w * w)])
    W = cons(cen)
    dW = torch.empty((15, W.shape[1]), dtype=torch.float64, device=W.device)
    h = 1e-6
    for i in range(3):
        e = torch.zeros(3, dtype=torch.float64, device=W.device)
        e[i] = h
        dW[i::3] = (cons(cen + e) - cons(cen - e)) / (2 * h)
    return W.contiguous(), dW


def _adjoint_inputs(case, seed, W):
    """Adjoint of the step's result and the frozen step, as the reverse
    sweep of a gradient run has them."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    lW = torch.randn(W.shape, generator=g, dtype=torch.float64).to(W.device)
    ldW = (0.05 * torch.randn((15, W.shape[1]), generator=g, dtype=torch.float64)).to(W.device)
    dt = 0.02 / max(case["nx"], case["ny"], case["nz"]) * (10.0 if case["problem"] == "vortex" else 1.0)
    return lW, ldW, dt


def prepare(case, seed):
    W, dW = _fields(case, seed)
    st = gks.State(_gks_mesh(*_key(case)), _params(case))
    s = dict(state=st, steps=case["steps"], call=case["call"], W=W, dW=dW, single=case["precision"] != 0)
    if case["problem"] == "sphere":
        st.set_fixed_state(W, dW)
    if case["call"] == "host":
        s["W"], s["dW"] = W.cpu().pin_memory(), dW.cpu().pin_memory()
        s["out"] = torch.empty_like(s["W"]).pin_memory(), torch.empty_like(s["dW"]).pin_memory()
    if case["call"] == "adjoint":
        s["lam"] = _adjoint_inputs(case, seed, W)
    return s


def run(s):
    st = s["state"]
    if s["call"] == "host":
        return st.step_host(s["W"], s["dW"], s["steps"], 0.0, *s["out"])
    if s["call"] == "adjoint":
        lW, ldW, dt = s["lam"]
        return st.adjoint_step(s["W"], s["dW"], lW, ldW, dt)
    st.init(s["W"], s["dW"])
    st.step(s["steps"])
    W, dW = st.get()
    if s["single"]:
        # an FP32-bulk run carries FP32 results; its caller keeps them so
        return W.float(), dW.float()
    return W, dW


def work(case):
    """Bytes: the state read and written once, the stencil operators and the
    face geometry read once.  Flops: about 2,000 for the kinetic solution at
    a Gauss point and 2,500 for a cell's reconstruction, in each stage."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["problem"] == "batch":
        rng = np.random.Generator(np.random.PCG64(1000 * nx + 10 * ny + nz))
        nc = 6 * int((rng.integers(nx, ny + 1, size=case["members"]) ** 3).sum())
    elif case["problem"] == "sphere":
        nc = 6 * nx * (ny - 2) * nz + 3 * nx * 2 * nz
    else:
        nc = 6 * nx * ny * nz
    real = 4 if case["precision"] == 1 else 8
    op = 156 * real + 2 * 22 * (8 if case["precision"] == 0 else 4)
    flops = 2 * nc * (6 * 2000 + 2500)
    if case["call"] == "adjoint":
        return {"bytes": nc * (4 * 160 + op), "flops": 3 * flops}
    return {"bytes": nc * (2 * 160 + op), "flops": case["steps"] * flops}


# ------------------------------------------------------- the exact result --
# The method in FP64 torch operations.  Fields are component lists over
# cells or faces; local face f of a cell is opposite to its vertex f.

_PAIRS = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]


class _Geometry:
    def __init__(self, mesh):
        v = _vertices(mesh)
        dev = v.device
        nc = v.shape[0]
        tet = torch.as_tensor(mesh["tet"], device=dev)
        self.nc, self.dev = nc, dev
        self.case = torch.as_tensor(mesh["case"], device=dev).long() if "case" in mesh else None
        self.ncase = int(mesh.get("ncase", 1))
        self.vol = torch.linalg.det(v[:, 1:] - v[:, :1]).abs() / 6.0
        cen = v.mean(1)
        d = v - cen[:, None]
        self.mom = torch.stack([(d[..., i] * d[..., j]).sum(1) / 20.0 for i, j in _PAIRS], 1)  # [nc, 6]
        # the three vertices of each local face, by ascending id
        other = torch.tensor([[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]], device=dev)
        ids = tet[:, other]                                   # [nc, 4, 3]
        order = ids.argsort(-1)
        ids = ids.gather(-1, order)
        pos = d[:, other].gather(2, order[..., None].expand(-1, -1, -1, 3))
        nv = int(tet.max()) + 1
        key = ((ids[..., 0] * nv + ids[..., 1]) * nv + ids[..., 2]).reshape(-1)
        key, half = key.sort(stable=True)
        first = torch.ones_like(key, dtype=torch.bool)
        first[1:] = key[1:] != key[:-1]
        face = first.cumsum(0) - 1
        nf = int(face[-1]) + 1
        self.nf = nf
        lh = half[first]
        rh = torch.full((nf,), -1, device=dev, dtype=torch.long)
        rh[face[~first]] = half[~first]
        self.L, self.R = lh // 4, torch.where(rh >= 0, rh // 4, rh)
        pos = pos.reshape(-1, 3, 3)
        w = torch.full((3, 3), 1.0 / 6.0, device=dev, dtype=torch.float64)
        w += 0.5 * torch.eye(3, device=dev, dtype=torch.float64)
        self.XL = torch.einsum("ka,fad->fkd", w, pos[lh])
        self.XR = torch.einsum("ka,fad->fkd", w, pos[rh.clamp_min(0)])
        tri = pos[lh]
        an = 0.5 * torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0])
        an = an * torch.sign((an * tri.mean(1)).sum(1))[:, None]  # out of the left cell
        self.area = an.norm(dim=1)
        self.n = an / self.area[:, None]
        self.kind = torch.zeros(nf, dtype=torch.long, device=dev)
        if mesh.get("bkind") is not None:
            self.kind = torch.as_tensor(mesh["bkind"], device=dev).reshape(-1).long()[lh]
        # cell -> faces: id, sign, neighbour, offset of its centroid, Gauss points
        fid = torch.empty(nc * 4, dtype=torch.long, device=dev)
        fid[half] = face
        self.fid = fid.reshape(nc, 4)
        left = self.L[self.fid] == torch.arange(nc, device=dev)[:, None]
        self.sign = torch.where(left, 1.0, -1.0).double()
        self.nb = torch.where(left, self.R[self.fid], self.L[self.fid])
        off = (self.XL - self.XR).mean(1)                     # right centroid in the left cell's frame
        self.off = off[self.fid] * self.sign[..., None]       # [nc, 4, 3]
        self.G = torch.where(left[..., None, None], self.XL[self.fid], self.XR[self.fid])  # [nc, 4, 3, 3]
        self.dr = 3.0 * self.vol / self.area[self.fid].sum(1)


def _basis(x, mom):
    """The nine zero-mean basis functions at offsets x [..., 3]."""
    return torch.cat([x] + [(x[..., i] * x[..., j] - mom[..., p])[..., None] for p, (i, j) in enumerate(_PAIRS)], -1)


def _solve_ls(rows, eq, here):
    """min |rows a - r|^2 with eq a = e (rows of eq where `here`): the
    operator [n, unknowns, r + e] by the normal equations' saddle system."""
    n, m, u = rows.shape
    q = eq.shape[1]
    A = torch.zeros((n, u + q, u + q), dtype=rows.dtype, device=rows.device)
    B = torch.zeros((n, u + q, m + q), dtype=rows.dtype, device=rows.device)
    eq = eq * here[..., None]
    A[:, :u, :u] = rows.transpose(1, 2) @ rows
    A[:, u:, :u] = eq
    A[:, :u, u:] = eq.transpose(1, 2)
    A[:, range(u, u + q), range(u, u + q)] = 1.0 - here
    B[:, :u, :m] = rows.transpose(1, 2)
    B[:, range(u, u + q), range(m, m + q)] = here
    return torch.linalg.solve(A, B)[:, :u]


class _Stencils:
    """P1 slopes b = M1 dQ and P2 coefficients a = M2 [dQ; grad], in
    coordinates of the cell's own size; at constrained walls the momenta's
    operators W1, W2 with the cell average as one more datum."""

    def __init__(self, g, case, chunk=150_000):
        has = (g.nb >= 0).double()
        h = g.vol ** (1.0 / 3.0)
        pw = torch.cat([h[:, None].expand(-1, 3), (h * h)[:, None].expand(-1, 6)], 1)  # scale of the unknowns
        self.M1, self.M2 = torch.empty((g.nc, 3, 4), dtype=torch.float64, device=g.dev), torch.empty(
            (g.nc, 9, 16), dtype=torch.float64, device=g.dev)
        wall = ((g.nb < 0) & (g.kind[g.fid] == NOSLIP)) if case["constraint"] else None
        self.wall = wall.any(1).nonzero()[:, 0] if wall is not None else torch.zeros(0, dtype=torch.long, device=g.dev)
        eye = torch.eye(3, dtype=torch.float64, device=g.dev)

        def parts(c):
            hc = h[c][:, None, None]
            d = g.off[c] / hc
            nb = g.nb[c].clamp_min(0)
            own = g.mom[c] / (hc[:, 0] ** 2)
            other = g.mom[nb] / (hc ** 2)
            avg = _basis(d, own[:, None] - other)                     # neighbour averages of the basis
            grad = torch.zeros((len(c), 4, 3, 9), dtype=torch.float64, device=g.dev)
            grad[..., :3] = eye
            for p, (i, j) in enumerate(_PAIRS):
                grad[:, :, i, 3 + p] += d[..., j]
                grad[:, :, j, 3 + p] += d[..., i]
            return d, own, avg, (grad * has[c][:, :, None, None]).reshape(len(c), 12, 9)

        def put(c, x):
            """columns: gradient data carry one power of h"""
            x = x / pw[c][:, :, None]
            return torch.cat([x[..., 12:16], x[..., :12] * h[c][:, None, None], x[..., 16:]], -1)
        for s in range(0, g.nc, chunk):
            c = torch.arange(s, min(s + chunk, g.nc), device=g.dev)
            d, own, avg, grad = parts(c)
            self.M2[c] = put(c, _solve_ls(grad, avg, has[c]))
            rows = d * has[c][..., None]
            self.M1[c] = torch.linalg.solve(rows.transpose(1, 2) @ rows, rows.transpose(1, 2)) / h[c][:, None, None]
            if not case["weno"] and case["order"] == 3:
                # boundary cells: the least-squares linear fit to the same data
                e = (has[c].sum(1) < 4).nonzero()[:, 0]
                if len(e):
                    r = torch.cat([rows[e], (eye * has[c][e][:, :, None, None]).reshape(len(e), 12, 3)], 1)
                    x = torch.linalg.solve(r.transpose(1, 2) @ r, r.transpose(1, 2)) / h[c][e][:, None, None]
                    self.M2[c[e]] = 0.0
                    self.M2[c[e], :3, :4] = x[..., :4]
                    self.M2[c[e], :3, 4:] = x[..., 4:] * h[c][e][:, None, None]
        if len(self.wall):
            c = self.wall
            d, own, avg, grad = parts(c)
            on = wall[c].double()
            gp = g.G[c] / h[c][:, None, None, None]
            eq = torch.cat([avg, _basis(gp, own[:, None, None]).reshape(len(c), 12, 9)], 1)
            here = torch.cat([has[c], on.repeat_interleave(3, 1)], 1)
            x = _solve_ls(grad, eq, here)
            x = torch.cat([x[..., :16], -x[..., 16:].sum(-1, keepdim=True)], -1)
            self.W2 = put(c, x)
            y = _solve_ls(d * has[c][..., None], gp.mean(2), on)
            self.W1 = torch.cat([y[..., :4], -y[..., 4:].sum(-1, keepdim=True)], -1) / h[c][:, None, None]


def _reconstruct(g, st, case, W, dW):
    """R of every cell: [5][nc, 10] about the centroid (constant, x, y, z,
    xx, xy, xz, yy, yz, zz)."""
    has = (g.nb >= 0).double()
    nb = g.nb.clamp_min(0)
    v23, v43 = (g.vol ** (2.0 / 3.0)), (g.vol ** (4.0 / 3.0))
    eps = 1e-8
    out = []
    for q in range(5):
        Q = W[q]
        dq = (Q[nb] - Q[:, None]) * has
        data = torch.cat([dq, (dW[3 * q:3 * q + 3].T[nb] * has[..., None]).reshape(g.nc, 12)], 1)
        a = torch.einsum("ckj,cj->ck", st.M2, data)
        b = torch.einsum("cij,cj->ci", st.M1, dq)
        if len(st.wall) and 1 <= q <= 3:
            c = st.wall
            a = a.index_put((c,), torch.einsum("ckj,cj->ck", st.W2, torch.cat([data[c], Q[c][:, None]], 1)))
            b = b.index_put((c,), torch.einsum("cij,cj->ci", st.W1, torch.cat([dq[c], Q[c][:, None]], 1)))
        if not case["weno"]:
            r = a if case["order"] == 3 else torch.cat([b, torch.zeros_like(a[:, 3:])], 1)
        else:
            b1 = v23 * (b * b).sum(1)
            bj = v23[:, None] * (b[nb] ** 2).sum(-1)
            nn = has.sum(1)
            tot = 0.0
            for i in range(4):
                for j in range(i):
                    tot = tot + (bj[:, i] - bj[:, j]).abs() * has[:, i] * has[:, j]
            s1 = (tot / (nn * (nn - 1) / 2)) ** (4.0 / 3.0)
            w1 = (1.0 + s1[:, None] / (eps + bj)) * has
            b0 = (w1 * bj).sum(1) / w1.sum(1)
            if case["order"] == 2:
                s = (b1 - b0).abs() ** (4.0 / 3.0)
                w0, w1 = (1 + (s / (eps + b0)) ** 2) / 11, (1 + (s / (eps + b1)) ** 2) * 10 / 11
                r = torch.cat([(w1 / (w0 + w1) * 1.1)[:, None] * b, torch.zeros_like(a[:, 3:])], 1)
            else:
                H = torch.stack([2 * a[:, 3], a[:, 4], a[:, 5], a[:, 4], 2 * a[:, 6], a[:, 7], a[:, 5], a[:, 7],
                                 2 * a[:, 8]], 1).reshape(-1, 3, 3)
                m = g.mom
                M = torch.stack([m[:, 0], m[:, 1], m[:, 2], m[:, 1], m[:, 3], m[:, 4], m[:, 2], m[:, 4], m[:, 5]],
                                1).reshape(-1, 3, 3)
                first = (a[:, :3] ** 2).sum(1) + torch.einsum("cli,cij,clj->c", H, M, H)
                second = H[:, 0, 0] ** 2 + a[:, 4] ** 2 + a[:, 5] ** 2 + H[:, 1, 1] ** 2 + a[:, 7] ** 2 + H[:, 2, 2] ** 2
                b2 = v23 * first + v43 * second
                s = (0.5 * ((b2 - b1).abs() + (b2 - b0).abs())) ** (4.0 / 3.0)
                w0, w1, w2 = [gm * (1 + (s / (eps + be)) ** 2) / 111 for gm, be in ((1, b0), (10, b1), (100, b2))]
                c2 = w2 / (w0 + w1 + w2) * 1.11
                cb = w1 / (w0 + w1 + w2) * 1.1 - c2 * 0.099099099099099099
                r = torch.cat([c2[:, None] * a[:, :3] + cb[:, None] * b, c2[:, None] * a[:, 3:]], 1)
        c0 = Q - (r[:, 3:] * g.mom).sum(1)
        out.append(torch.cat([c0[:, None], r], 1))
    # cells with a non-positive density or pressure at a face Gauss point
    # fall back to their averages
    X = g.G.reshape(g.nc, 12, 3)
    val = [_eval(p[:, None], X)[0] for p in out]
    pr = val[4] - 0.5 * (val[1] ** 2 + val[2] ** 2 + val[3] ** 2) / val[0]
    ok = ((val[0] > 0) & (pr > 0)).all(1)
    return [torch.where(ok[:, None], p, torch.cat([W[q][:, None], torch.zeros_like(p[:, 1:])], 1))
            for q, p in enumerate(out)]


def _eval(p, X):
    """Value and gradient of R at offsets X."""
    x, y, z = X[..., 0], X[..., 1], X[..., 2]
    c = [p[..., k] for k in range(10)]
    v = (c[0] + c[1] * x + c[2] * y + c[3] * z + c[4] * x * x + c[5] * x * y + c[6] * x * z + c[7] * y * y
         + c[8] * y * z + c[9] * z * z)
    return v, (c[1] + 2 * c[4] * x + c[5] * y + c[6] * z, c[2] + c[5] * x + 2 * c[7] * y + c[8] * z,
               c[3] + c[6] * x + c[8] * y + 2 * c[9] * z)


# a polynomial in u, v, w and xi^2: {(powers): coefficient}
_PSI = [{(0, 0, 0, 0): 1.0}, {(1, 0, 0, 0): 1.0}, {(0, 1, 0, 0): 1.0}, {(0, 0, 1, 0): 1.0},
        {(2, 0, 0, 0): 0.5, (0, 2, 0, 0): 0.5, (0, 0, 2, 0): 0.5, (0, 0, 0, 1): 0.5}]
_ONE = _PSI[0]
_VEL = _PSI[1:4]


def _times(*ps):
    out = {(0, 0, 0, 0): 1.0}
    for p in ps:
        new = {}
        for a, x in out.items():
            for b, y in p.items():
                k = tuple(i + j for i, j in zip(a, b))
                new[k] = new.get(k, 0.0) + x * y
        out = new
    return out


class _Maxwellian:
    """rho, U, lambda of a state (face frame) and its velocity moments, over
    the whole space or the half space u sign > 0."""

    def __init__(self, W, half=0):
        self.rho = W[0]
        self.U = [W[1] / W[0], W[2] / W[0], W[3] / W[0]]
        self.p = (GAMMA - 1) * (W[4] - 0.5 * (W[1] * self.U[0] + W[2] * self.U[1] + W[3] * self.U[2]))
        self.lam = 0.5 * self.rho / self.p
        h = 0.5 / self.lam
        self.tab = []
        for i in range(3):
            m = [torch.ones_like(h), self.U[i]]
            if i == 0 and half:
                s = self.lam.sqrt() * self.U[0]
                m[0] = 0.5 * torch.special.erfc(-half * s)
                m[1] = self.U[0] * m[0] + half * 0.5 / math.sqrt(math.pi) * torch.exp(-s * s) / self.lam.sqrt()
            for k in range(5):
                m.append(self.U[i] * m[k + 1] + (k + 1) * h * m[k])
            self.tab.append(m)
        self.tab.append([torch.ones_like(h), K_INT * h, (K_INT * K_INT + 2 * K_INT) * h * h])

    def mean(self, poly):
        out = 0.0
        for (i, j, k, l), c in poly.items():
            t = c * self.tab[0][i]
            for n, e in ((1, j), (2, k), (3, l)):
                if e:
                    t = t * self.tab[n][e]
            out = out + t
        return out

    def psi(self, extra):
        """rho <psi extra>"""
        return [self.rho * self.mean(_times(p, extra)) for p in _PSI]

    def slope(self, dW):
        """a of a . psi = d ln g along dW"""
        dU = [(dW[1 + i] - self.U[i] * dW[0]) / self.rho for i in range(3)]
        u2 = sum(u * u for u in self.U)
        dp = (GAMMA - 1) * (dW[4] - sum(u * d for u, d in zip(self.U, dW[1:4])) + 0.5 * u2 * dW[0])
        dl = 0.5 * (dW[0] - self.rho * dp / self.p) / self.p
        a = [dW[0] / self.rho + 0.5 * (K_INT + 3) * dl / self.lam - dl * u2
             - 2 * self.lam * sum(u * d for u, d in zip(self.U, dU))]
        return a + [2 * self.lam * d + 2 * u * dl for u, d in zip(self.U, dU)] + [-2 * dl]

    def apsi(self, a, extra):
        """rho <psi (a . psi) extra>"""
        return [self.rho * sum(a[m] * self.mean(_times(_PSI[k], _PSI[m], extra)) for m in range(5)) for k in range(5)]


def _sum5(*terms):
    return [sum(c * x[k] for c, x in terms) for k in range(5)]


def _point(case, L, gL, R, gR, dt):
    """The kinetic solution at Gauss points, face frame: int_0^{dt/2} F,
    int_0^dt F - twice that, W(0), W(dt) - W(0)."""
    mu, prandtl = _mu(case), 0.72 if case["problem"] == "sphere" else 1.0
    sides, zero = [], 0.0
    for W, g, half in ((L, gL, 1), (R, gR, -1)):
        m = _Maxwellian(W, half)
        a = [m.slope(g[i]) for i in range(3)]
        sides.append((m, a, W))
    Wc = _sum5(*[(1.0, m.psi(_ONE)) for m, _, _ in sides])
    C = _Maxwellian(Wc)
    dWc = [_sum5(*[(1.0, m.apsi(a[i], _ONE)) for m, a, _ in sides]) for i in range(3)]
    ac = [C.slope(dWc[i]) for i in range(3)]
    conv = lambda m, a, extra: _sum5(*[(1.0, m.apsi(a[i], _times(_VEL[i], extra))) for i in range(3)])  # noqa: E731
    rate = [-x for x in conv(C, ac, _ONE)]
    Ac = C.slope(rate)
    tau = mu / C.p if case["viscous"] else torch.zeros_like(C.p)
    pl, pr = sides[0][0].p, sides[1][0].p
    tn = (tau if case["viscous"] else 0.01 * dt) + ((pl - pr) / (pl + pr)).abs() * dt
    U1 = _VEL[0]

    def kinetic(t0):
        """integrals over [0, t0] of e^{-t/tn} and t e^{-t/tn}"""
        e = torch.exp(-t0 / tn)
        return tn * (1 - e), tn * (tn * (1 - e) - t0 * e)

    f0, f1 = C.psi(U1), conv(C, ac, U1)
    f2 = C.apsi(Ac, U1)
    side = []
    for m, a, W in sides:
        s0, s1, w1 = m.psi(U1), conv(m, a, U1), conv(m, a, _ONE)
        s2 = w2 = None
        if case["viscous"]:
            full = _Maxwellian(W)
            A = full.slope([-x for x in conv(full, a, _ONE)])
            s2, w2 = m.apsi(A, U1), m.apsi(A, _ONE)
        side.append((s0, s1, s2, m.psi(_ONE), w1, w2))

    def integral(t0, state):
        """int_0^t0 of the flux (or of the state)"""
        e0, e1 = kinetic(t0)
        q1, q2, q3 = t0 - e0, e1 + tau * e0 - tau * t0, 0.5 * t0 * t0 - tau * t0 + tau * e0
        if state:
            out = _sum5((q1, Wc), (q2 - q3, [-x for x in rate]))
        else:
            out = _sum5((q1, f0), (q2, f1), (q3, f2))
        for s in side:
            x0, x1, x2 = s[3:] if state else s[:3]
            out = _sum5((1.0, out), (e0, x0), (-(tau * e0 + e1), x1))
            if x2 is not None:
                out = _sum5((1.0, out), (-tau * e0, x2))
        return out

    Fh, F = integral(0.5 * dt, False), integral(dt, False)
    if case["viscous"] and prandtl != 1.0:
        for f, t0 in ((Fh, 0.5 * dt), (F, dt)):
            s = integral(t0, True)
            q = [y[4] - sum(u * v for u, v in zip(C.U, y[1:4])) + 0.5 * sum(u * u for u in C.U) * y[0] for y in (f, s)]
            f[4] = f[4] + (1.0 / prandtl - 1.0) * (q[0] - C.U[0] * q[1])
    # W(t) at t = 0 and t = dt; a . u and A moments of the equilibrium cancel
    E = torch.exp(-dt / tn)
    w0, wt = Wc, _sum5((1.0 - E, Wc), ((dt + tau) * E - tau, [-x for x in rate]), (dt - tau + tau * E, rate))
    for s in side:
        w0 = _sum5((1.0, w0), (-tau, s[4]))
        wt = _sum5((1.0, wt), (E, s[3]), (-(tau + dt) * E, s[4]))
        if s[5] is not None:
            w0 = _sum5((1.0, w0), (-tau, s[5]))
            wt = _sum5((1.0, wt), (-tau * E, s[5]))
    return Fh, _sum5((1.0, F), (-2.0, Fh)), w0, _sum5((1.0, wt), (-1.0, w0))


def _face_sums(g, case, W, R, dt, fixed, chunk):
    """Per face: sum over its Gauss points of weight times (Fh, D, W0, dWt),
    global frame: four [5, nf]."""
    tot = [[], [], [], []]
    for s in range(0, g.nf, chunk):
        f = slice(s, min(s + chunk, g.nf))
        n, kind, nf = g.n[f], g.kind[f], g.n[f].shape[0]
        hasr = (g.R[f] >= 0)[:, None].expand(nf, 3)
        # an orthonormal frame about the normal
        e = torch.eye(3, dtype=n.dtype, device=n.device)[n.abs().argmin(1)]
        t1 = torch.linalg.cross(n, e)
        t1 = t1 / t1.norm(dim=1, keepdim=True)
        T = torch.stack([n, t1, torch.linalg.cross(n, t1)], 1)  # rows

        def rot(v, M):
            """momenta of a component list by M [nf, 3, 3]"""
            return [v[0]] + [sum(M[:, j, i][:, None] * v[1 + i] for i in range(3)) for j in range(3)] + [v[4]]

        def side(cell, X):
            v = [_eval(R[q][cell][:, None], X) for q in range(5)]
            grad = [[sum(T[:, j, i][:, None] * v[q][1][i] for i in range(3)) for q in range(5)] for j in range(3)]
            return rot([x[0] for x in v], T), [rot(x, T) for x in grad]
        L, gL = side(g.L[f], g.XL[f])
        rc = g.R[f].clamp_min(0)
        Rr, gR = side(rc, g.XR[f])
        bnd = g.R[f] < 0
        if bool(bnd.any()):
            k = kind[:, None].expand(nf, 3)
            neg = lambda x, idx: [-y if i in idx else y for i, y in enumerate(x)]  # noqa: E731
            zero = torch.zeros_like(L[0])
            own = rot([W[q][g.L[f]][:, None].expand(nf, 3) for q in range(5)], T)
            ghosts = {OPEN: (own, [[zero] * 5] * 3),
                      SLIP: (neg(L, (1,)), [neg(gL[0], (0, 2, 3, 4)), neg(gL[1], (1,)), neg(gL[2], (1,))]),
                      NOSLIP: (neg(L, (1, 2, 3)), [neg(x, (0, 4)) for x in gL])}
            if fixed is not None:
                W0, dW0 = fixed
                c = g.L[f]
                gg = [[dW0[3 * q + i][c][:, None].expand(nf, 3) for q in range(5)] for i in range(3)]
                val = [W0[q][c][:, None] + sum(gg[i][q] * g.XL[f][..., i] for i in range(3)) for q in range(5)]
                ghosts[FIXED] = (rot(val, T), [rot([sum(T[:, j, i][:, None] * gg[i][q] for i in range(3))
                                                    for q in range(5)], T) for j in range(3)])
            for b, (gw, gg) in ghosts.items():
                m = ~hasr & (k == b)
                Rr = [torch.where(m, x, y) for x, y in zip(gw, Rr)]
                gR = [[torch.where(m, x, y) for x, y in zip(a, c)] for a, c in zip(gg, gR)]
        dtf = dt if g.case is None else dt[g.case[g.L[f]]][:, None]
        got = _point(case, L, gL, Rr, gR, dtf)
        w = g.area[f][:, None] / 3.0
        for t, x in zip(tot, got):
            t.append(torch.stack([(w * y).sum(1) for y in rot(x, T.transpose(1, 2))]))
    return [torch.cat(t, 1) for t in tot]


def _exact_step(g, st, case, W, dW, dt, fixed=None, chunk=400_000):
    gather = lambda x: (x[:, g.fid] * g.sign).sum(-1)                                       # noqa: E731
    spread = lambda x: torch.stack([(x[q][g.fid][..., None] * g.sign[..., None] * g.n[g.fid]).sum(1)  # noqa: E731
                                    for q in range(5)]).permute(0, 2, 1).reshape(15, g.nc)
    Fh, D, w0, wt = _face_sums(g, case, W, _reconstruct(g, st, case, W, dW), dt, fixed, chunk)
    Ws = W - gather(Fh) / g.vol
    S = gather(2.0 * Fh - D / 3.0)
    dWs, G = spread(w0 + 0.5 * wt) / g.vol, spread(w0)
    _, D, _, wt = _face_sums(g, case, Ws, _reconstruct(g, st, case, Ws, dWs), dt, fixed, chunk)
    return W - (S + gather(4.0 / 3.0 * D)) / g.vol, (G + spread(wt)) / g.vol


def _time_step(g, case, W):
    u = (W[1] ** 2 + W[2] ** 2 + W[3] ** 2).sqrt() / W[0]
    p = (GAMMA - 1) * (W[4] - 0.5 * W[0] * u * u)
    d = g.dr / (u + (GAMMA * p / W[0]).sqrt())
    if case["viscous"]:
        d = torch.minimum(d, g.dr ** 2 * W[0] / (3 * _mu(case)))
    if g.case is None:
        return 0.5 * d.min()
    return 0.5 * torch.full((g.ncase,), math.inf, dtype=d.dtype, device=d.device).scatter_reduce(0, g.case, d, "amin")


def exact(case, seed):
    W, dW = _fields(case, seed)
    g = _Geometry(_mesh(*_key(case)))
    st = _Stencils(g, case)
    if case["call"] == "adjoint":
        lW, ldW, dt = _adjoint_inputs(case, seed, W)
        W.requires_grad_(True)
        dW.requires_grad_(True)
        nW, ndW = _exact_step(g, st, case, W, dW, torch.tensor(dt, dtype=torch.float64, device=W.device))
        return torch.autograd.grad((nW * lW).sum() + (ndW * ldW).sum(), (W, dW))
    fixed = (W, dW) if case["problem"] == "sphere" else None
    with torch.no_grad():
        for _ in range(case["steps"]):
            W, dW = _exact_step(g, st, case, W, dW, _time_step(g, case, W), fixed)
    return W, dW
