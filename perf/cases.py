"""What a user of this framework has it do, as measurable cases: single steps and
solves of each preconditioner, the reverse step, a fit sample through autograd, a
forward rollout, the learned preconditioner's training step, the recurrent pressure
solver, the volumetric initialisation, the APIC transfers and the splatting
renderer, each through the calls a program makes (``fluidstep``, ``rollout``,
``volume_init``), at sizes from this repository's configurations, tests and
benchmark.

``prepare`` makes inputs on the GPU from the seed alone; ``exact`` restates each
case's mathematics in 64 bits on dense staggered arrays, without the library.

Array conventions: dense cell arrays are (nz, ny, nx), x fastest; component c of a
MAC field has one more entry along axis c; the library layout is (nz + 1, ny + 1,
pitch), pitch = nx + 1 rounded up to a multiple of 4.
"""
import math

import numpy as np
import torch

from paper_2503_00868_gb300 import apic as AP
from paper_2503_00868_gb300 import fluidstep as F
from paper_2503_00868_gb300 import rollout as RO
from paper_2503_00868_gb300 import train_percnn as TP
from paper_2503_00868_gb300 import train_precond as TC
from paper_2503_00868_gb300 import volume_init as VI

AIR, LIQUID, SOLID = 0, 1, 2
DT = 1.0 / 30.0
STREAM = (0.9, 0.0, 0.4)  # a river across the grid's axes
PRECOND = {"jacobi": F.FS_PRECOND_JACOBI, "mic0": F.FS_PRECOND_MIC0, "mg": F.FS_PRECOND_MG,
           "learned_mg": F.FS_PRECOND_LEARNED_MG}


def listed():
    return [
        # the smallest simulation: one forward step in a closed 32^3 box full of liquid with
        # MIC(0); launches, host reads and the wavefront's latency
        {"name": "step_mic0_32", "kind": "step", "scene": "full", "nx": 32, "ny": 32, "nz": 32, "precond": "mic0"},
        # one forward step with the default preconditioner on a ragged grid, as a first user
        # without any option set runs it
        {"name": "step_jacobi_odd", "kind": "step", "scene": "blob", "nx": 101, "ny": 75, "nz": 90,
         "precond": "jacobi"},
        # one forward and one reverse step with multigrid on a small ragged grid: the inner loop of
        # a low-resolution fit, where V-cycle launches and latencies count
        {"name": "adjoint_mg_small_odd", "kind": "adjoint", "scene": "blob", "nx": 53, "ny": 44, "nz": 39,
         "precond": "mg"},
        # the headline: one forward and one reverse step at 256^3 with multigrid
        {"name": "adjoint_mg_256", "kind": "adjoint", "scene": "blob", "nx": 256, "ny": 256, "nz": 256,
         "precond": "mg"},
        # one sample of a fit at a quarter of the full fit's cells: river scene with inflow, loss on the
        # surface band, gradients to the viscosity and the initial field through autograd
        {"name": "fit_sample_river", "kind": "fit", "scene": "river", "nx": 128, "ny": 64, "nz": 128,
         "precond": "mg", "frames": 1, "upwind": False},
        # a forward rollout at 128^3, as targets and re-simulations are made
        {"name": "rollout_mg_128", "kind": "rollout", "scene": "blob", "nx": 128, "ny": 128, "nz": 128,
         "precond": "mg", "frames": 4},
        # projection of a strongly divergent field on a union of spheres with the learned
        # preconditioner in front of the V-cycle (network inference)
        {"name": "project_learned_256", "kind": "project", "scene": "spheres", "nx": 256, "ny": 256, "nz": 256,
         "precond": "learned_mg"},
        # a training step of the learned preconditioner on a 64^3 pair: network forward, backward, Adam
        {"name": "train_net_64", "kind": "train", "scene": "spheres", "nx": 64, "ny": 64, "nz": 64},
        # projection by the recurrent convolutional solver, 100 sub-steps
        {"name": "project_percnn_128", "kind": "percnn", "scene": "blob", "nx": 128, "ny": 128, "nz": 128,
         "substeps": 100},
        # volumetric initialisation of the full fit's grid: wall profile and 200 constrained projections
        {"name": "volume_init_192", "kind": "volume", "scene": "river", "nx": 192, "ny": 128, "nz": 192,
         "iters": 200},
        # particle <-> grid transfers of a re-simulation at 256^3, four particles per liquid cell
        {"name": "apic_256", "kind": "apic", "scene": "blob", "nx": 256, "ny": 256, "nz": 256, "ppc": 4},
        # a 1920 x 1080 frame of the Gaussians of a 128^3 blob, one per liquid cell
        {"name": "splat_1080p", "kind": "splat", "scene": "blob", "nx": 128, "ny": 128, "nz": 128,
         "width": 1920, "height": 1080, "degree": 0},
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "adjoint", "fit", "rollout", "project", "train", "percnn", "volume", "apic", "splat"])
    hi = {"step": 160, "adjoint": 224, "fit": 144, "rollout": 144, "project": 224, "train": 96, "percnn": 192,
          "volume": 192, "apic": 192, "splat": 160}[kind]
    case = {"kind": kind, "nx": _size(rng, 24, hi), "ny": _size(rng, 24, hi), "nz": _size(rng, 24, hi)}
    case["scene"] = {"fit": "river", "volume": "river", "train": "spheres"}.get(kind, "blob")
    if kind == "step":
        case["precond"] = rng.choice(["jacobi", "mic0", "mg"])
        case["scene"] = rng.choice(["blob", "full", "river"])
    elif kind == "adjoint":
        case["precond"] = "mg"
        case["scene"] = rng.choice(["blob", "river"])
    elif kind == "fit":
        case["precond"] = "mg"
        # several frames only with the upwind reverse of convection: the exact reverse has the kinks of
        # the trilinear sample, and two runs whose states differ in the last bits fall on either side
        case["upwind"] = rng.random() < 0.5
        case["frames"] = rng.randint(2, 4) if case["upwind"] else 1
    elif kind == "rollout":
        case["precond"] = "mg"
        case["frames"] = rng.randint(2, 5)
    elif kind == "project":
        case["precond"] = rng.choice(["jacobi", "mg", "learned_mg"])
        case["scene"] = rng.choice(["blob", "spheres"])
    elif kind == "percnn":
        case["substeps"] = _size(rng, 10, 120)
    elif kind == "volume":
        case["iters"] = _size(rng, 20, 200)
    elif kind == "apic":
        case["ppc"] = rng.randint(1, 8)
    elif kind == "splat":
        case["width"], case["height"] = _size(rng, 160, 1920), _size(rng, 120, 1080)
        case["degree"] = rng.randint(0, 3)
    return case


# ---- inputs --------------------------------------------------------------------

def _shapes(c):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    return (nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx)


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 64 + stream)
    return g


def _blur(a, sigma=3.0, radius=9):
    """Separable Gaussian, clamp to edge."""
    w = [math.exp(-0.5 * (x / sigma) ** 2) for x in range(-radius, radius + 1)]
    for axis in range(3):
        n = a.shape[axis]
        out = torch.zeros_like(a)
        for x, wx in zip(range(-radius, radius + 1), w):
            idx = torch.arange(n, device=a.device).add_(x).clamp_(0, n - 1)
            out += (wx / sum(w)) * a.index_select(axis, idx)
        a = out
    return a


def _noise(c, seed, stream, blur=True):
    """N(0, 1) per MAC component, blurred over 3 cells, wall-normal faces zero; or unblurred."""
    g = _gen(seed, stream)
    out = [torch.randn(s, generator=g, device="cuda") for s in _shapes(c)]
    if blur:
        out = [_blur(a) for a in out]
        for a, axis in zip(out, (2, 1, 0)):
            a.select(axis, 0).zero_()
            a.select(axis, a.shape[axis] - 1).zero_()
    return out


def _centres(c):
    """Cell-centre indices (k, j, i) + 1/2, broadcastable."""
    ar = [torch.arange(n, device="cuda", dtype=torch.float64) + 0.5 for n in (c["nz"], c["ny"], c["nx"])]
    return ar[0].view(-1, 1, 1), ar[1].view(1, -1, 1), ar[2].view(1, 1, -1)


def _scene(c, seed):
    """(types uint8 (nz, ny, nx) on the GPU, dense fixed-face values or None)."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    k, j, i = _centres(c)
    if c["scene"] == "full":
        return torch.full((nz, ny, nx), LIQUID, dtype=torch.uint8, device="cuda"), None
    # particle arrays have one length whatever the seed
    rng = np.random.default_rng(0 if c["kind"] == "apic" else seed)
    if c["scene"] == "spheres":
        n = min(nx, ny, nz)
        for _ in range(1000):
            inside = torch.zeros((nz, ny, nx), dtype=torch.bool, device="cuda")
            for r, p in zip(rng.uniform(20, 60, 8) * n / 256.0, rng.uniform(0, 1, (8, 3))):
                inside |= (i - p[0] * nx) ** 2 + (j - p[1] * ny) ** 2 + (k - p[2] * nz) ** 2 <= r * r
            # ragged boxes hold the same spheres in more room
            if 0.15 * n ** 3 <= float(inside.sum()) <= 0.5 * n ** 3:
                break
        return torch.where(inside, LIQUID, AIR).to(torch.uint8), None
    # an ellipsoid resting on the floor, about 40 % of the box
    a, cc = rng.uniform(0.40, 0.49, 2)
    b = min(0.40 * 3.0 / (4.0 * math.pi * a * cc), 0.49)
    inside = ((i / nx - 0.5) / a) ** 2 + ((j / ny - b) / b) ** 2 + ((k / nz - 0.5) / cc) ** 2 <= 1.0
    types = torch.where(inside, LIQUID, AIR).to(torch.uint8)
    if c["scene"] == "blob":
        return types, None
    low = (j < 0.25 * ny).expand(nz, ny, nx)  # a river: a layer of a quarter of the height, inflow at x = 0
    types = torch.where(low, LIQUID, types).to(torch.uint8)
    bc = [torch.zeros(s, device="cuda") for s in _shapes(c)]
    bc[0][:, :, 0] = 0.5 * ((types[:, :, 0] == LIQUID) & low[:, :, 0])
    return types, bc


def _pair(c, types, seed):
    """A (right-hand side, pressure) pair L_p q = b on the liquid, smooth and rough parts as CG residuals have."""
    shape = (c["nz"], c["ny"], c["nx"])
    n = torch.randn(shape, generator=_gen(seed, 9), device="cuda")
    q = (8.0 * _blur(n) + 0.2 * n).double() * (types == LIQUID)
    b = _Ref(c, types, None).poisson(q)
    return b.float(), q.float()


def _particles(c, types, seed):
    """`ppc` jittered particles per liquid cell, in cell order, with velocities and affine matrices."""
    dx, ppc = 1.0 / c["ny"], c["ppc"]
    g = _gen(seed, 11)
    kji = torch.nonzero(types == LIQUID)
    cell = kji[:, [2, 1, 0]].float().repeat_interleave(ppc, 0)
    n = cell.shape[0]
    x = (cell + torch.rand((n, 3), generator=g, device="cuda")) * dx
    p = AP.Particles(x, torch.full((n,), 1.0 / ppc, device="cuda"),
                     (torch.eye(3, device="cuda") * (0.3 * dx) ** 2).reshape(1, 9).repeat(n, 1))
    p.v = 0.2 * torch.randn((n, 3), generator=g, device="cuda")
    p.C = 2.0 * torch.randn((n, 9), generator=g, device="cuda")
    return p


def _cloud(c, types, seed):
    """One Gaussian per liquid cell: position, opacity, covariance, spherical-harmonic colour; a camera around it."""
    dx, g = 1.0 / c["ny"], _gen(seed, 13)
    kji = torch.nonzero(types == LIQUID)
    n = kji.shape[0]
    rand = lambda *s: torch.rand(s, generator=g, device="cuda")  # noqa: E731
    x = (kji[:, [2, 1, 0]].float() + 0.5 + 0.5 * (rand(n, 3) - 0.5)) * dx
    q = torch.randn((n, 4), generator=g, device="cuda")
    w, a, b, d = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    Q = torch.stack([1 - 2 * (b * b + d * d), 2 * (a * b - w * d), 2 * (a * d + w * b),
                     2 * (a * b + w * d), 1 - 2 * (a * a + d * d), 2 * (b * d - w * a),
                     2 * (a * d - w * b), 2 * (b * d + w * a), 1 - 2 * (a * a + b * b)], 1).view(n, 3, 3)
    s = (0.3 + 0.6 * rand(n, 3)) * dx
    A = torch.bmm(Q * (s * s).unsqueeze(1), Q.transpose(1, 2)).reshape(n, 9).contiguous()
    sh = 0.3 * torch.randn((n, (c["degree"] + 1) ** 2, 3), generator=g, device="cuda")
    rng = np.random.default_rng(seed)
    ex, ez = c["nx"] * dx, c["nz"] * dx
    target, radius = np.array([0.5 * ex, 0.2, 0.5 * ez]), 1.6 * max(1.0, ex, ez)
    az, el = rng.uniform(0, 2 * math.pi), rng.uniform(0.1, 0.6)
    fwd = -np.array([math.cos(el) * math.sin(az), math.sin(el), math.cos(el) * math.cos(az)])
    right = np.cross(fwd, [0.0, 1.0, 0.0])
    right /= np.linalg.norm(right)
    R = np.stack([right, np.cross(fwd, right), fwd])
    f = 0.5 * c["height"] / math.tan(0.4)
    cam = F.make_camera(R, -R @ (target - radius * fwd), f, f, 0.5 * c["width"], 0.5 * c["height"], c["width"],
                        c["height"], 0.01, (0.1, 0.2, 0.3))
    return x.contiguous(), 0.3 + 0.65 * rand(n), A, sh, cam


def _params(c):
    kw = dict(dx=1.0 / c["ny"], dt=DT, nu=0.01, g=(0.0, -9.81, 0.0), maxit_p=20000, maxit_v=4000)
    kw["precond"] = PRECOND[c.get("precond", "jacobi")]
    if c["kind"] == "percnn":
        kw["pressure_solver"] = F.FS_SOLVER_PERCNN
    if c.get("upwind"):
        kw["advect_grad"] = F.FS_ADVECT_GRAD_UPWIND
    return kw


def _speed(c, seed):
    return torch.tensor(VI.synthetic_surface_speed(c["nx"], c["nz"], seed), dtype=torch.float32,
                        device="cuda").contiguous()


def prepare(case, seed):
    c = dict(case)
    types, bc = _scene(c, seed)
    kind = c["kind"]
    grid = F.Grid(c["nx"], c["ny"], c["nz"], **_params(c))
    s = {"case": c, "grid": grid}
    if kind != "splat":
        grid.set_mask(types, grid.pack(bc) if bc is not None else None)
    if kind in ("step", "adjoint", "fit", "rollout"):
        s["u"] = grid.pack([a + (0 if bc is None else b) for a, b in zip(_noise(c, seed, 0), bc or [0, 0, 0])])
    if kind in ("step", "adjoint"):
        s["out"], s["uv"], s["gin"] = grid.zeros(), grid.zeros(), grid.zeros()
    if kind == "adjoint":
        s["target"], s["g"] = grid.pack(_noise(c, seed, 1)), grid.zeros()
    if kind == "fit":
        s["targets"] = {c["frames"]: grid.pack(_noise(c, seed, 2))}
        s["leaves"] = [t.requires_grad_(True) for t in s["u"]]
        s["nu"] = torch.tensor(0.01, requires_grad=True)
    if kind in ("project", "percnn"):
        s["u"], s["out"], s["q"] = grid.pack(_noise(c, seed, 3, blur=kind == "percnn")), grid.zeros(), grid.empty_cell()
        if kind == "percnn":
            F.fs_percnn_load(grid.ctx, TP.default_kernel(), c["substeps"])
        elif c["precond"] == "learned_mg":
            F.fs_net_load(grid.ctx, TC.role_weights("net_mg"))
    if kind == "train":
        F.fs_net_load(grid.ctx, TC.role_weights("net"))
        s["b"], s["q"] = (grid.empty_cell() for _ in range(2))
        for t, a in zip((s["b"], s["q"]), _pair(c, types, seed)):
            t[: c["nz"], : c["ny"], : c["nx"]] = a
    if kind == "volume":
        s["vinf"] = _speed(c, seed)
    if kind == "apic":
        s["p"] = _particles(c, types, seed)
        s["v"], s["C"], s["x"], s["F"] = (torch.empty_like(t) for t in (s["p"].v, s["p"].C, s["p"].x, s["p"].F))
        s["A"] = torch.empty_like(s["p"].A)
        s["u"] = grid.zeros()
    if kind == "splat":
        s["cloud"] = _cloud(c, types, seed)
        s["rgb"] = torch.empty((c["height"], c["width"], 3), device="cuda")
        s["T"] = torch.empty((c["height"], c["width"]), device="cuda")
    return s


# ---- one pass ------------------------------------------------------------------

def run(s):
    c, grid = s["case"], s["grid"]
    kind = c["kind"]
    if kind == "step":
        grid.step(s["u"], s["out"], s["uv"])
        return {"u": list(s["out"]), "visc": list(s["uv"])}
    if kind == "adjoint":
        grid.step(s["u"], s["out"], s["uv"])
        for g, o, t in zip(s["g"], s["out"], s["target"]):  # the cotangent of |u - t|^2 / 2
            torch.sub(o, t, out=g)
        _, gnu, _ = grid.adjoint_step(s["u"], s["g"], s["gin"], s["uv"])
        return {"u": list(s["out"]), "g_in": list(s["gin"]), "g_nu": gnu}
    if kind == "fit":
        for t in s["leaves"] + [s["nu"]]:
            t.grad = None
        loss = RO.rollout_loss(grid, F.Mac(*s["leaves"]), s["nu"], c["frames"], s["targets"], 2, alpha=0.1)
        loss.backward()
        return {"loss": float(loss.detach()), "g_nu": s["nu"].grad, "g_u": [t.grad for t in s["leaves"]]}
    if kind == "rollout":
        return [list(m) for m in RO.forward_states(grid, s["u"], c["frames"])[1:]]
    if kind in ("project", "percnn"):
        for d, u in zip(s["out"], s["u"]):  # the projection works in place: a copy of the field to project
            d.copy_(u)
        grid.project(s["out"], s["q"])
        return {"u": list(s["out"]), "q": s["q"]}
    if kind == "train":
        loss = F.fs_net_grad(grid.ctx, s["b"], s["q"])
        grad = F.fs_net_grad_read(grid.ctx)
        F.fs_net_adam(grid.ctx, 1e-5, 1)
        return {"loss": loss, "grad": grad}
    if kind == "volume":
        u, n0, n1 = VI.volume_init(grid, STREAM, s["vinf"], 0.1, c["iters"], 0.5 * c["ny"] ** 2)
        return {"u": list(u), "div": [n0, n1]}
    if kind == "apic":
        p, dx = s["p"], 1.0 / c["ny"]
        s["x"].copy_(p.x)  # the transfers move the particles in place: the re-simulation's initial state
        s["F"].copy_(p.F)
        F.fs_p2g(grid.ctx, p.x, p.v, p.C, p.m, s["u"])
        F.fs_g2p(grid.ctx, s["x"], s["v"], s["C"], s["u"], F=s["F"], A0=p.A0, A_out=s["A"], dt=DT, advance=True,
                 lo=1.5 * dx, hi=max(c["nx"], c["ny"], c["nz"]) * dx)
        return {"u": list(s["u"]), "x": s["x"], "v": s["v"], "C": s["C"], "F": s["F"], "A": s["A"]}
    x, op, A, sh, cam = s["cloud"]
    F.fs_splat_render_sh(grid.ctx, x, op, A, sh, c["degree"], cam, s["rgb"], s["T"])
    return {"rgb": s["rgb"], "T": s["T"]}


def work(case):
    """Inputs read once, outputs written once, and the operations that the call's own arguments fix (sub-steps,
    iterations, network layers); a solve to a tolerance counts one operator apply."""
    c, kind = case, case["kind"]
    cells = c["nx"] * c["ny"] * c["nz"]
    field = 12.0 * cells
    occ = {"full": 1.0, "spheres": 0.2, "blob": 0.4, "river": 0.55}[c["scene"]]
    if kind == "step":
        return {"bytes": 3 * field + cells, "flops": 150.0 * occ * cells}
    if kind == "adjoint":
        return {"bytes": 5 * field + cells, "flops": 400.0 * occ * cells}
    if kind == "fit":
        return {"bytes": 3 * field + cells, "flops": 550.0 * occ * cells * c["frames"]}
    if kind == "rollout":
        return {"bytes": (1 + c["frames"]) * field + cells, "flops": 150.0 * occ * cells * c["frames"]}
    layers = 2.0 * 27 * (2 * 16 + 3 * 16 * 16 + 16)  # flops per cell of one network pass
    if kind == "project":
        return {"bytes": 2 * field + 5 * cells, "flops": (30.0 + (layers if c["precond"] == "learned_mg" else 0)) * occ * cells}
    if kind == "percnn":
        return {"bytes": 2 * field + 5 * cells, "flops": (c["substeps"] * 70.0 + 30) * occ * cells}
    if kind == "train":
        return {"bytes": 9.0 * cells, "flops": 3.0 * layers * cells}
    if kind == "volume":
        return {"bytes": field + 5 * cells, "flops": c["iters"] * 35.0 * occ * cells}
    if kind == "apic":
        n = occ * cells * c["ppc"]
        return {"bytes": n * 4.0 * (16 + 21 + 33) + field, "flops": n * 81.0 * 20}
    n = occ * cells
    return {"bytes": n * 4.0 * (13 + 3 * (c["degree"] + 1) ** 2) + 16.0 * c["width"] * c["height"],
            "flops": n * 300.0}


# ---- the same in 64 bits ---------------------------------------------------------

def _shift(a, axis, d):
    """a moved by d along axis, zeros shifted in: out[i] = a[i + d]."""
    out = torch.zeros_like(a)
    n = a.shape[axis]
    if d > 0:
        out.narrow(axis, 0, n - d).copy_(a.narrow(axis, d, n - d))
    else:
        out.narrow(axis, -d, n + d).copy_(a.narrow(axis, 0, n + d))
    return out


def _cg(apply, inv_diag, b, x=None):
    """Jacobi-preconditioned CG in 64 bits to 1e-13."""
    x = torch.zeros_like(b) if x is None else x.clone()
    r = b - apply(x)
    z = inv_diag * r
    p, rz, stop = z.clone(), (r * z).sum(), 1e-26 * (b * b).sum()
    for it in range(20000):
        if it % 50 == 0 and float((r * r).sum()) <= float(stop):
            break
        q = apply(p)
        a = rz / (p * q).sum().clamp_min(1e-300)
        x += a * p
        r -= a * q
        z = inv_diag * r
        new = (r * z).sum()
        p = z + (new / rz.clamp_min(1e-300)) * p
        rz = new
    return x


class _Ref:
    """The fluid step on dense staggered float64 arrays (component c along axis 2 - c)."""

    def __init__(self, c, types, bc, nu=0.01):
        self.dx, self.nu, self.n = 1.0 / c["ny"], nu, (c["nx"], c["ny"], c["nz"])
        self.dt, self.g = DT, (0.0, -9.81, 0.0)
        self.liq, self.air = types == LIQUID, types == AIR
        pad = torch.full([n + 2 for n in types.shape], SOLID, dtype=torch.uint8, device=types.device)
        pad[1:-1, 1:-1, 1:-1] = types
        self.bc = [torch.zeros(s, dtype=torch.float64, device=types.device) if bc is None else b.double()
                   for s, b in zip(_shapes(c), bc or [0, 0, 0])]
        self.fluid, self.fixed, self.lo, self.hi = [], [], [], []
        for comp in range(3):
            ax = 2 - comp
            inner = [slice(1, -1)] * 3
            inner[ax] = slice(None)
            t = pad[tuple(inner)]
            lo, hi = t.narrow(ax, 0, t.shape[ax] - 1), t.narrow(ax, 1, t.shape[ax] - 1)
            fixed = (lo == SOLID) | (hi == SOLID)
            self.fixed.append(fixed)
            self.fluid.append(~fixed & ((lo == LIQUID) | (hi == LIQUID)))
            self.lo.append(lo)
            self.hi.append(hi)
        open_ = (self.liq | self.air).double()
        self.diag = sum(_shift(open_, ax, d) for ax in range(3) for d in (-1, 1)) * self.liq
        near_air = sum(_shift(self.air.double(), ax, d) for ax in range(3) for d in (-1, 1)) > 0
        self.band = self.liq & near_air
        self.singular = not bool(self.band.any())

    def poisson(self, q):
        nb = sum(_shift(q, ax, d) for ax in range(3) for d in (-1, 1))
        return (self.diag * q - nb) * self.liq

    def divergence(self, u):
        return sum(a.narrow(2 - k, 1, a.shape[2 - k] - 1) - a.narrow(2 - k, 0, a.shape[2 - k] - 1)
                   for k, a in enumerate(u)) / self.dx

    def rhs(self, u):
        b = -self.dx * self.dx * self.divergence(u) * self.liq
        return b - (b.sum() / self.liq.sum()) * self.liq if self.singular else b

    def grad(self, q):
        """(q_hi - q_lo) / dx on fluid faces."""
        out = []
        for k in range(3):
            ax = 2 - k
            z = torch.zeros_like(q.narrow(ax, 0, 1))
            p = torch.cat([z, q, z], ax)
            d = p.narrow(ax, 1, p.shape[ax] - 1) - p.narrow(ax, 0, p.shape[ax] - 1)
            out.append(torch.where(self.fluid[k], d / self.dx, torch.zeros_like(d)))
        return out

    def project(self, u):
        inv = torch.where(self.diag > 0, 1.0 / self.diag.clamp_min(1.0), torch.zeros_like(self.diag))
        q = _cg(self.poisson, inv, self.rhs(u))
        if self.singular:
            q = q - (q.sum() / self.liq.sum()) * self.liq
        return [a - d for a, d in zip(u, self.grad(q))], q

    def viscosity(self, u, dirichlet):
        cc, out = self.nu * self.dt / self.dx ** 2, []
        for k in range(3):
            fl = self.fluid[k]
            cnt = (fl | self.fixed[k]).double()
            n = sum(_shift(cnt, ax, d) for ax in range(3) for d in (-1, 1))
            diag = 1.0 + cc * n

            def apply(v):
                return (diag * v - cc * sum(_shift(v, ax, d) for ax in range(3) for d in (-1, 1))) * fl

            b = u[k] * fl
            if dirichlet:
                fv = self.bc[k] * self.fixed[k]
                b = b + cc * sum(_shift(fv, ax, d) for ax in range(3) for d in (-1, 1)) * fl
            out.append(_cg(apply, fl / diag, b, u[k] * fl))
        return out

    def advect(self, u):
        """Back-traced components with the body force on fluid faces, zero elsewhere."""
        mean = [0.5 * (a.narrow(2 - k, 0, a.shape[2 - k] - 1) + a.narrow(2 - k, 1, a.shape[2 - k] - 1))
                for k, a in enumerate(u)]
        out = []
        for k in range(3):
            shape, fl = u[k].shape, self.fluid[k]
            at = torch.nonzero(fl)
            lin = (at[:, 0] * shape[1] + at[:, 1]) * shape[2] + at[:, 2]
            s, base = [], []
            for e in range(3):
                if e == k:
                    v = u[k].reshape(-1)[lin]
                else:
                    low = at.clone()
                    low[:, 2 - k] -= 1
                    m = mean[e]
                    flat = lambda a: m.reshape(-1)[(a[:, 0] * m.shape[1] + a[:, 1]) * m.shape[2] + a[:, 2]]  # noqa: E731
                    v = 0.5 * (flat(low) + flat(at))
                n = shape[2 - e]
                p = (at[:, 2 - e].double() - self.dt / self.dx * v).clamp(0.0, n - 1.0)
                b = p.detach().floor().clamp(0, n - 2)
                s.append(p - b)
                base.append(b.long())
            val = 0.0
            for dz in (0, 1):
                for dy in (0, 1):
                    for dx in (0, 1):
                        w = 1.0
                        for f, d in zip(s, (dx, dy, dz)):
                            w = w * (f if d else 1.0 - f)
                        val = val + w * u[k].reshape(-1)[((base[2] + dz) * shape[1] + base[1] + dy) * shape[2] + base[0] + dx]
            out.append(torch.zeros(shape.numel(), dtype=torch.float64, device=lin.device).index_put(
                (lin,), val + self.dt * self.g[k]).reshape(shape))
        return out

    def compose(self, v):
        return [torch.where(f, a, torch.where(x, b, torch.zeros_like(a)))
                for a, f, x, b in zip(v, self.fluid, self.fixed, self.bc)]

    def step(self, u):
        uv = self.compose(self.viscosity(self.advect(u), True))
        return self.project(uv)[0], uv

    def adjoint(self, u, uv, g):
        """(dL/du, dL/dnu) for the cotangent g of the step's output."""
        x = self.viscosity(self.project([a * f for a, f in zip(g, self.fluid)])[0], False)
        leaf = [a.detach().clone().requires_grad_(True) for a in u]
        sum((a * b).sum() for a, b in zip(self.advect(leaf), x)).backward()
        return [a.grad for a in leaf], self.nu_grad(uv, x)

    def loss(self, u, t, alpha, beta):
        total = 0.0
        nb = sum(int((f & (self._at(self.band, k, 0) | self._at(self.band, k, 1))).sum()) for k, f in enumerate(self.fluid))
        for k, f in enumerate(self.fluid):
            m = f & (self._at(self.band, k, 0) | self._at(self.band, k, 1))
            total = total + beta / (2.0 * nb) * ((u[k] - t[k]) ** 2 * m).sum()
        mid = lambda w: [0.5 * (a.narrow(2 - k, 0, a.shape[2 - k] - 1) + a.narrow(2 - k, 1, a.shape[2 - k] - 1))[self.band]  # noqa: E731
                         for k, a in enumerate(w)]
        a, b = mid(u), mid(t)
        norm = lambda v: torch.sqrt(sum(x * x for x in v) + 1e-16)  # noqa: E731
        cos = sum(x * y for x, y in zip(a, b)) / (norm(a) * norm(b))
        return total + alpha / int(self.band.sum()) * (1.0 - cos).sum()

    def _at(self, cells, k, side):
        """A cell mask on the faces of component k: the face's low (0) or high (1) cell."""
        ax = 2 - k
        z = torch.zeros_like(cells.narrow(ax, 0, 1))
        return torch.cat([z, cells], ax) if side == 0 else torch.cat([cells, z], ax)

    def loss_grad(self, u, t, alpha, beta):
        leaf = [a.detach().clone().requires_grad_(True) for a in u]
        v = self.loss(leaf, t, alpha, beta)
        v.backward()
        return float(v.detach()), [a.grad for a in leaf]

    def adjoint_upwind(self, u, uv, g):
        """adjoint() with the upwind surrogate of the reverse of convection."""
        x = self.viscosity(self.project([a * f for a, f in zip(g, self.fluid)])[0], False)
        conv = self.compose(self.advect(u))
        out = [a.clone() for a in x]
        mean = [0.5 * (a.narrow(2 - k, 0, a.shape[2 - k] - 1) + a.narrow(2 - k, 1, a.shape[2 - k] - 1))
                for k, a in enumerate(u)]
        for k in range(3):
            ax = 2 - k
            for e in range(3):
                ae = 2 - e
                if e == k:
                    vel = u[k]
                else:
                    edge = lambda m, i: m.narrow(ax, i, 1)  # noqa: E731
                    m = mean[e]
                    m = torch.cat([edge(m, 0), m, edge(m, m.shape[ax] - 1)], ax)
                    vel = 0.5 * (m.narrow(ax, 0, m.shape[ax] - 1) + m.narrow(ax, 1, m.shape[ax] - 1))
                idx = torch.arange(conv[k].shape[ae], device=vel.device).view([-1 if i == ae else 1 for i in range(3)])
                back = (conv[k] - _shift(conv[k], ae, -1)) * (idx > 0)
                ahead = (_shift(conv[k], ae, 1) - conv[k]) * (idx < conv[k].shape[ae] - 1)
                gv = -self.dt / self.dx * torch.where(vel > 0, back, ahead) * x[k] * self.fluid[k]
                if e == k:
                    out[k] += gv
                    continue
                # the face's two cells, and the two faces of component e at each
                cell = 0.25 * (gv.narrow(ax, 0, gv.shape[ax] - 1) + gv.narrow(ax, 1, gv.shape[ax] - 1))
                out[e].narrow(ae, 0, out[e].shape[ae] - 1).add_(cell)
                out[e].narrow(ae, 1, out[e].shape[ae] - 1).add_(cell)
        return out, self.nu_grad(uv, x)

    def nu_grad(self, uv, x):
        dot = 0.0
        for k in range(3):
            cnt = self.fluid[k] | self.fixed[k]
            n = sum(_shift(cnt.double(), ax, d) for ax in range(3) for d in (-1, 1))
            lu = n * uv[k] - sum(_shift(uv[k] * cnt, ax, d) for ax in range(3) for d in (-1, 1))
            dot += float((x[k] * lu * self.fluid[k]).sum())
        return -self.dt * dot / self.dx ** 2


def _embed(c, dense):
    """Dense arrays in the library layout, zeros in the padding."""
    out = []
    for a in dense:
        t = torch.zeros((c["nz"] + 1, c["ny"] + 1, (c["nx"] + 4) // 4 * 4), dtype=torch.float64, device=a.device)
        t[: a.shape[0], : a.shape[1], : a.shape[2]] = a
        out.append(t)
    return out


def _exact_fit(c, ref, u, target):
    states, viscs = [u], []
    for _ in range(c["frames"]):
        out, uv = ref.step(states[-1])
        states.append(out)
        viscs.append(uv)
    loss, g = ref.loss_grad(states[-1], target, 0.1, 1.0)
    gnu = 0.0
    for n in range(c["frames"] - 1, -1, -1):
        g, d = (ref.adjoint_upwind if c["upwind"] else ref.adjoint)(states[n], viscs[n], g)
        gnu += d
    return {"loss": loss, "g_nu": gnu, "g_u": _embed(c, g)}


def _exact_volume(c, ref, vinf):
    dx, free, u = ref.dx, [], []
    col = vinf.double().unsqueeze(1)  # (nz, 1, nx)
    for k, (f, x) in enumerate(zip(ref.fluid, ref.fixed)):
        j = torch.arange(f.shape[1], device="cuda", dtype=torch.float64).view(1, -1, 1)
        y = (j if k == 1 else j + 0.5) * dx
        r = (y / 0.1).clamp(0.0, 1.0)
        fac = torch.where(r >= 1.0, torch.ones_like(r), 1.5 * r - 0.5 * r ** 3)
        v = col
        if k != 1:
            ax = 2 - k
            v = torch.cat([v.narrow(ax, 0, 1), v, v.narrow(ax, v.shape[ax] - 1, 1)], ax)
            v = 0.5 * (v.narrow(ax, 0, v.shape[ax] - 1) + v.narrow(ax, 1, v.shape[ax] - 1))
        main = STREAM[k] * v * fac
        u.append(torch.where(f, main.expand(f.shape), ref.bc[k] * x))
        surface = ((ref.lo[k] == LIQUID) & (ref.hi[k] == AIR)) | ((ref.lo[k] == AIR) & (ref.hi[k] == LIQUID))
        free.append(f & ~surface)
    n = sum(m.narrow(2 - k, 0, m.shape[2 - k] - 1).double() + m.narrow(2 - k, 1, m.shape[2 - k] - 1).double()
            for k, m in enumerate(free))
    eps = 0.5 * c["ny"] ** 2
    div = lambda: ref.divergence(u) * ref.liq  # noqa: E731
    n0 = float(div().norm())
    for _ in range(c["iters"]):
        lam = -div() / (n / dx ** 2 + eps)
        for k in range(3):
            ax = 2 - k
            z = torch.zeros_like(lam.narrow(ax, 0, 1))
            p = torch.cat([z, lam, z], ax)
            d = p.narrow(ax, 0, p.shape[ax] - 1) - p.narrow(ax, 1, p.shape[ax] - 1)
            u[k] = u[k] + torch.where(free[k], d / dx, torch.zeros_like(d))
    return {"u": _embed(c, u), "div": [n0, float(div().norm())]}


def _nodes(x, comp, dx):
    """Base node and quadratic B-spline weights of component `comp` around positions x."""
    base, w = [], []
    for a in range(3):
        s = x[:, a] / dx - (0.0 if a == comp else 0.5)
        b = (s - 0.5).floor()
        f = s - b
        base.append(b.long())
        w.append((0.5 * (1.5 - f) ** 2, 0.75 - (f - 1.0) ** 2, 0.5 * (f - 0.5) ** 2))
    return base, w


def _exact_apic(c, p):
    dx = 1.0 / c["ny"]
    f64 = lambda t: t.double()  # noqa: E731
    shapes, n = _shapes(c), p.x.shape[0]
    u, parts = [], [slice(a, min(a + (1 << 22), n)) for a in range(0, n, 1 << 22)]
    for comp in range(3):
        shape = shapes[comp]
        size = shape[0] * shape[1] * shape[2]
        mv, ms = torch.zeros((2, size), dtype=torch.float64, device="cuda")
        for sl in parts:
            x, m = f64(p.x[sl]), f64(p.m[sl])
            for lin, wt, d in _walk(x, comp, dx, shape):
                val = f64(p.v[sl, comp]) + sum(f64(p.C[sl, 3 * comp + a]) * d[a] for a in range(3))
                mv.index_add_(0, lin, wt * m * val)
                ms.index_add_(0, lin, wt * m)
        u.append(torch.where(ms > 0, mv / ms.clamp_min(1e-300), torch.zeros_like(mv)).view(shape))
    out = {k: [] for k in "xvCFA"}
    for sl in parts:
        x = f64(p.x[sl])
        v, C = torch.zeros_like(x), torch.zeros((x.shape[0], 3, 3), dtype=torch.float64, device="cuda")
        for comp in range(3):
            for lin, wt, d in _walk(x, comp, dx, shapes[comp]):
                wu = wt * u[comp].reshape(-1)[lin]
                v[:, comp] += wu
                for a in range(3):
                    C[:, comp, a] += 4.0 / dx ** 2 * wu * d[a]
        Fn = f64(p.F[sl]).view(-1, 3, 3)
        Fn = Fn + DT * torch.bmm(C, Fn)
        out["x"].append((x + DT * v).clamp(1.5 * dx, max(c["nx"], c["ny"], c["nz"]) * dx))
        out["v"].append(v)
        out["C"].append(C.view(-1, 9))
        out["F"].append(Fn.view(-1, 9))
        out["A"].append(torch.bmm(torch.bmm(Fn, f64(p.A0[sl]).view(-1, 3, 3)), Fn.transpose(1, 2)).reshape(-1, 9))
    return {"u": _embed(c, u), **{k: torch.cat(v) for k, v in out.items()}}


def _walk(x, comp, dx, shape):
    """(flat node, weight, node - particle) of the 27 nodes; nodes outside the array get weight zero."""
    base, w = _nodes(x, comp, dx)
    for kz in range(3):
        for ky in range(3):
            for kx in range(3):
                idx = [base[0] + kx, base[1] + ky, base[2] + kz]
                ok = torch.ones_like(base[0], dtype=torch.bool)
                for a in range(3):
                    ok &= (idx[a] >= 0) & (idx[a] < shape[2 - a])
                lin = torch.where(ok, (idx[2] * shape[1] + idx[1]) * shape[2] + idx[0], torch.zeros_like(idx[0]))
                d = [(idx[a].double() + (0.0 if a == comp else 0.5)) * dx - x[:, a] for a in range(3)]
                yield lin, w[0][kx] * w[1][ky] * w[2][kz] * ok, d


def _sh_basis(deg, d):
    """Real spherical harmonics of degree <= 3 of unit vectors, in the order l^2 + l + m."""
    x, y, z = d.unbind(1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 * math.sqrt(1 / pi))]
    if deg >= 1:
        a = math.sqrt(3 / (4 * pi))
        Y += [-a * y, a * z, -a * x]
    if deg >= 2:
        b, e = math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi))
        Y += [b * x * y, -b * y * z, e * (2 * z * z - x * x - y * y), -b * x * z, 0.5 * b * (x * x - y * y)]
    if deg >= 3:
        f, g = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi))
        h, k = math.sqrt(21 / (32 * pi)), math.sqrt(7 / (16 * pi))
        Y += [-f * y * (3 * x * x - y * y), g * x * y * z, -h * y * (4 * z * z - x * x - y * y),
              k * z * (2 * z * z - 3 * x * x - 3 * y * y), -h * x * (4 * z * z - x * x - y * y),
              0.5 * g * z * (x * x - y * y), -f * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _exact_splat(c, cloud):
    x, op, A, sh, cam = cloud
    dev = x.device
    t64 = lambda v: torch.tensor(np.asarray(v, np.float32), device=dev).double()  # noqa: E731
    R, t, bg = t64(list(cam.R)).view(3, 3), t64(list(cam.t)), t64(list(cam.bg))
    fx, fy, cx, cy = (float(np.float32(v)) for v in (cam.fx, cam.fy, cam.cx, cam.cy))
    W, H, TILE = c["width"], c["height"], 16
    xc = x.double() @ R.T + t
    X, Y, Z = xc.unbind(1)
    mx, my = fx * X / Z + cx, fy * Y / Z + cy
    zero = torch.zeros_like(Z)
    J = torch.stack([fx / Z, zero, -fx * X / Z ** 2, zero, fy / Z, -fy * Y / Z ** 2], 1).view(-1, 2, 3)
    M = J @ R
    S = M @ A.double().view(-1, 3, 3) @ M.transpose(1, 2)
    det = S[:, 0, 0] * S[:, 1, 1] - S[:, 0, 1] * S[:, 1, 0]
    d = x.double() + (R.T @ t)
    col = (0.5 + torch.einsum("nj,njk->nk", _sh_basis(c["degree"], d / d.norm(dim=1, keepdim=True)),
                              sh.double())).clamp_min(0.0)
    con = torch.stack([S[:, 1, 1], -S[:, 0, 1], S[:, 0, 0]], 1) / det.unsqueeze(1)
    ex, ey = 3 * S[:, 0, 0].sqrt(), 3 * S[:, 1, 1].sqrt()
    ok = (Z > 0.01) & (det > 0)
    ntx, nty = -(-W // TILE), -(-H // TILE)
    x0, x1 = ((mx - ex) / TILE).floor().clamp(0, ntx).long(), ((mx + ex) / TILE).floor().clamp(-1, ntx - 1).long() + 1
    y0, y1 = ((my - ey) / TILE).floor().clamp(0, nty).long(), ((my + ey) / TILE).floor().clamp(-1, nty - 1).long() + 1
    wx, wy = (x1 - x0).clamp_min(0) * ok, (y1 - y0).clamp_min(0) * ok
    order = torch.argsort(Z.float(), stable=True)  # depth, ties by index
    cnt = (wx * wy)[order]
    gid = order.repeat_interleave(cnt)
    k = torch.arange(gid.numel(), device=dev) - (cnt.cumsum(0) - cnt).repeat_interleave(cnt)
    tile = (y0[gid] + k // wx[gid].clamp_min(1)) * ntx + x0[gid] + k % wx[gid].clamp_min(1)
    tile, perm = torch.sort(tile, stable=True)
    gid = gid[perm]
    per = torch.bincount(tile, minlength=ntx * nty)
    start = per.cumsum(0) - per
    rgb = bg.view(1, 1, 3).repeat(nty * TILE, ntx * TILE, 1)
    Tf = torch.ones((nty * TILE, ntx * TILE), dtype=torch.float64, device=dev)
    pix = torch.arange(TILE * TILE, device=dev)
    busy = torch.argsort(per, descending=True)
    busy = busy[: int((per > 0).sum())].tolist()
    counts = per.tolist()
    a = 0
    while a < len(busy):
        m = counts[busy[a]]
        b = a + max(1, min(len(busy) - a, (1 << 25) // (m * 256)))
        tl = torch.tensor(busy[a:b], device=dev)
        q = torch.arange(m, device=dev)
        valid = q.view(1, -1) < per[tl].view(-1, 1)
        ids = gid[torch.where(valid, start[tl].view(-1, 1) + q, torch.zeros_like(q))]
        px = ((tl % ntx) * TILE).view(-1, 1) + pix % TILE
        py = ((tl // ntx) * TILE).view(-1, 1) + pix // TILE
        ddx = px.double().view(-1, 1, 256) + 0.5 - mx[ids].unsqueeze(2)
        ddy = py.double().view(-1, 1, 256) + 0.5 - my[ids].unsqueeze(2)
        cn = con[ids].unsqueeze(3)
        md = cn[:, :, 0] * ddx ** 2 + 2 * cn[:, :, 1] * ddx * ddy + cn[:, :, 2] * ddy ** 2
        al = (op.double()[ids].unsqueeze(2) * torch.exp(-0.5 * md)).clamp_max(0.99)
        al = al * ((md <= 9) & (al >= 1.0 / 255) & valid.unsqueeze(2))
        after = torch.cumprod(1 - al, 1)
        al = al * (after >= 1e-4)  # the walk stops before the transmittance falls below 1e-4
        after = torch.cumprod(1 - al, 1)
        w = al * torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
        T = after[:, -1]
        Tf[py, px] = T
        rgb[py, px] = torch.einsum("tmp,tmc->tpc", w, col[ids]) + T.unsqueeze(2) * bg
        a = b
    return {"rgb": rgb[:H, :W].clone(), "T": Tf[:H, :W].clone()}


def _exact_train(c, types, b, q):
    """The energy-norm loss of the network (bf16 weights, inputs, activations and their gradients) and its gradient."""
    rnd = lambda t: t.to(torch.float32).to(torch.bfloat16).double()  # noqa: E731
    p = torch.tensor(TC.role_weights("net"), device="cuda").double()
    ch = [2, 16, 16, 16, 16, 1]
    W, B, at = [], [], 0
    for i in range(5):
        n = ch[i + 1] * ch[i] * 27
        W.append(rnd(p[at: at + n]).view(ch[i + 1], ch[i], 3, 3, 3))
        B.append(p[at + n: at + n + ch[i + 1]])
        at += n + ch[i + 1]
    taps = [(z, y, x) for z in range(3) for y in range(3) for x in range(3)]
    ref = _Ref(c, types, None)
    nz, ny, nx = types.shape
    b, q = b.double() * ref.liq, q.double() * ref.liq
    s = b.abs().max()
    pad = lambda t: torch.nn.functional.pad(t, (1, 1) * 3)  # noqa: E731
    win = lambda t, z, y, x: t[:, z: z + nz, y: y + ny, x: x + nx].reshape(t.shape[0], -1)  # noqa: E731
    code = torch.where(types == LIQUID, 1.0, torch.where(types == AIR, 0.0, -1.0)).double()
    a = [torch.stack([rnd((b / s) * ref.liq), code])]
    for i in range(5):
        src = pad(a[-1])
        o = sum(W[i][:, :, z, y, x] @ win(src, z, y, x) for z, y, x in taps) + B[i].view(-1, 1)
        o = o.view(-1, nz, ny, nx)
        a.append(rnd(o.clamp_min(0.0)) if i < 4 else o)
    tq = q / s
    e = (a[5][0] - tq) * ref.liq
    ae, den = ref.poisson(e), (tq * ref.poisson(tq)).sum()
    g = (2.0 / den * ae).unsqueeze(0)
    grads = [None] * 5
    for i in range(4, -1, -1):
        src, gf = pad(a[i]), g.reshape(g.shape[0], -1)
        gw = torch.stack([gf @ win(src, z, y, x).T for z, y, x in taps], 2)
        grads[i] = torch.cat([gw.reshape(-1), gf.sum(1)])
        if i:
            gp = pad(g)
            back = sum(W[i][:, :, 2 - z, 2 - y, 2 - x].T @ win(gp, z, y, x) for z, y, x in taps)
            g = rnd(back.view(-1, nz, ny, nx) * (a[i] > 0))
    return {"loss": float((e * ae).sum() / den), "grad": torch.cat(grads)}


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    cells = c["nx"] * c["ny"] * c["nz"]
    if kind in ("step", "adjoint", "fit", "rollout", "project") and cells > 5_000_000:
        return None  # the 64-bit solves would take over 20 seconds
    types, bc = _scene(c, seed)
    if kind == "splat":
        return _exact_splat(c, _cloud(c, types, seed))
    if kind == "apic":
        return _exact_apic(c, _particles(c, types, seed))
    if kind == "train":
        return _exact_train(c, types, *_pair(c, types, seed))
    ref = _Ref(c, types, bc)
    if kind == "volume":
        return _exact_volume(c, ref, _speed(c, seed))
    if kind in ("project", "percnn"):
        u = [a.double() for a in _noise(c, seed, 3, blur=kind == "percnn")]
        if kind == "project":
            v, q = ref.project(u)
        else:
            w = torch.tensor(np.asarray(TP.default_kernel(), np.float32), device="cuda").double().view(27)
            w = 0.5 * (w + w.flip(0))
            b, q = ref.rhs(u), torch.zeros(types.shape, dtype=torch.float64, device="cuda")
            nz, ny, nx = types.shape
            for _ in range(c["substeps"]):
                r = torch.nn.functional.pad((b - ref.poisson(q)) * ref.liq, (1, 1) * 3)
                q = q + sum(w[9 * z + 3 * y + x] * r[z: z + nz, y: y + ny, x: x + nx]
                            for z in range(3) for y in range(3) for x in range(3)) * ref.liq
            v = [a - d for a, d in zip(u, ref.grad(q))]
        return {"u": _embed(c, v), "q": _embed(c, [q])[0]}
    u = [(a + (0 if bc is None else b)).double() for a, b in zip(_noise(c, seed, 0), bc or [0, 0, 0])]
    if kind == "rollout":
        states = [u]
        for _ in range(c["frames"]):
            states.append(ref.step(states[-1])[0])
        return [_embed(c, s) for s in states[1:]]
    if kind == "fit":
        return _exact_fit(c, ref, u, [a.double() for a in _noise(c, seed, 2)])
    out, uv = ref.step(u)
    if kind == "step":
        return {"u": _embed(c, out), "visc": _embed(c, uv)}
    g, gnu = ref.adjoint(u, uv, [a - b.double() for a, b in zip(out, _noise(c, seed, 1))])
    return {"u": _embed(c, out), "g_in": _embed(c, g), "g_nu": gnu}
