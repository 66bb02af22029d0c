"""Performance cases: the calls a user of the library makes, over the range of their sizes.

A run of the library is a sequence of time steps; a step is a Newton-Krylov solve of the
Poisson-Nernst-Planck (PNP) block, with the Navier-Stokes (NS) block before it in a coupled
run.  The cases are the operators such a program calls on its own (residual, Jacobian
action in FP64, in FP32 and through a stored linearisation, NS matrix action), whole steps
(FP64, mixed precision, coupled), and the learned start's network (inference and training
gradient).  Meshes, parameters and boundary tables are those of the library's tests and
benchmark: uniform grids, octrees graded towards a membrane, random 2:1 octrees with
hanging nodes, periodic sides, 2D and 3D.

``exact`` evaluates the same weak form in 64 bits with torch alone: connectivity and
hanging constraints from the node coordinates, 2^d-point Gauss quadrature, the Jacobian
action by forward-mode differentiation, small nonlinear systems by dense Newton.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2301_05985_gb300 import pnp
from paper_2301_05985_gb300 import workloads as W

DEV = "cuda"
F64 = torch.float64
BDF2 = dict(beta0=1.5, beta1=-2.0, beta2=0.5)
K0, HID, NOUT = 216, 128, 3  # network: 216 -> 128 -> 128 -> 128 -> 3

# the Navier-Stokes block of the benchmark, converged two digits further so that the
# fields of a step do not depend on the path of the Krylov solver
NS_KW = dict(ns_Sc=1.0, ns_kappa=0.5, ns_mg_levels=8, mg_smooth=3, mg_omega=0.6, mg_coarse_its=32, ns_rtol=1e-10,
             ns_atol=1e-12, ns_fgmres=50)
MIXED_KW = dict(precision=pnp.PNP_F32, start_mode=pnp.PNP_START_EXTRAPOLATE, gmres_restart=60, gmres_max_it=3000,
                gmres_inner=24, dt_retries=2)
NEWTON_RTOL = 1e-10


def listed():
    return [
        # a 2D double-layer study on a laptop-sized grid: latency of one call
        dict(name="residual_2d_L5", kind="residual", mesh="uniform", dim=2, level=5, eps=0.05, dt=0.01, V=1.0, vel=0.0),
        # Newton's FP64 residual on the membrane-band octree of the benchmark, moving fluid
        dict(name="residual_band_L5_8", kind="residual", mesh="band", dim=3, level=5, fine=8, band=0.05, eps=1e-3,
             dt=1e-3, V=20.0, vel=0.5),
        # FP64 Jacobian action (the default solver's operator) on a uniform cube, Fourier velocity
        dict(name="jv64_L6", kind="jv64", mesh="uniform", dim=3, level=6, eps=1e-3, dt=1e-3, V=30.0, vel=0.1),
        # one FP32 Jacobian action at a new state (no stored linearisation), fluid at rest
        dict(name="jv32_band_L4_7", kind="jv32", mesh="band", dim=3, level=4, fine=7, band=0.05, eps=2e-3, dt=1e-3,
             V=20.0, vel=0.0),
        # the operator of the mixed-precision Krylov solves, on the benchmark's uniform cube
        dict(name="jv_linearized_L7", kind="jv_linearized", mesh="uniform", dim=3, level=7, eps=1e-3, dt=1e-3, V=30.0,
             vel=0.1),
        # the NS Krylov operator, FP64 (outer) and FP32 (preconditioner)
        dict(name="ns_matvec64_band_L5_8", kind="ns_matvec64", mesh="band", dim=3, level=5, fine=8, band=0.05, eps=1e-3,
             dt=1e-3, V=20.0, vel=0.5),
        dict(name="ns_matvec32_band_L4_7", kind="ns_matvec32", mesh="band", dim=3, level=4, fine=7, band=0.05, eps=2e-3,
             dt=1e-3, V=20.0, vel=0.5),
        # a time step with the library's default solver (FP64 GMRES, exact Newton), 2D
        dict(name="time_step_f64_2d_L5", kind="time_step", precision="f64", mesh="uniform", dim=2, level=5, eps=0.05,
             dt=0.01, V=5.0, vel=0.0),
        # a PNP time step in mixed precision on the small membrane-band octree
        dict(name="time_step_mixed_band_L4_7", kind="time_step", precision="mixed", mesh="band", dim=3, level=4, fine=7,
             band=0.05, eps=2e-3, dt=1e-3, V=20.0, vel=0.0),
        # the benchmark's step, NS then PNP, on the membrane-band octree
        dict(name="coupled_step_band_L5_8", kind="coupled_step", precision="mixed", mesh="band", dim=3, level=5, fine=8,
             band=0.05, eps=1e-3, dt=1e-3, V=20.0, vel=0.0),
        # the network on the nodes of a uniform level-5 cube, and one training gradient
        dict(name="mlp_forward_35937", kind="mlp_forward", rows=35937),
        dict(name="mlp_loss_grad_4096", kind="mlp_loss_grad", rows=4096),
    ]


def draw(rng):
    kind = rng.choice(["residual", "residual", "jv64", "jv32", "jv_linearized", "jv_linearized", "ns_matvec64",
                       "ns_matvec32", "time_step", "time_step", "coupled_step", "mlp_forward", "mlp_loss_grad"])
    if kind in ("mlp_forward", "mlp_loss_grad"):
        hi = 200000 if kind == "mlp_forward" else 65536
        return dict(kind=kind, rows=int(round(math.exp(rng.uniform(math.log(17), math.log(hi))))))
    if kind == "coupled_step":
        lv = rng.choice([3, 4])
        return dict(kind=kind, precision="mixed", mesh="band", dim=3, level=lv, fine=lv + 3,
                    band=round(rng.uniform(0.02, 0.08), 4), eps=round(rng.uniform(2e-3, 8e-3), 5),
                    dt=round(rng.uniform(5e-4, 1e-3), 6), V=round(rng.uniform(5.0, 20.0), 2), vel=0.0)
    if kind == "time_step" and rng.random() < 0.5:
        return dict(kind=kind, precision="f64", mesh="uniform", dim=2, level=rng.choice([4, 5]),
                    eps=round(rng.uniform(0.04, 0.1), 4), dt=round(rng.uniform(5e-3, 2e-2), 5),
                    V=round(rng.uniform(0.5, 6.0), 2), vel=0.0)
    if kind == "time_step":
        lv = rng.choice([3, 4])
        return dict(kind=kind, precision="mixed", mesh="band", dim=3, level=lv, fine=lv + rng.choice([2, 3]),
                    band=round(rng.uniform(0.02, 0.1), 4), eps=round(rng.uniform(2e-3, 1e-2), 5),
                    dt=round(rng.uniform(5e-4, 1e-3), 6), V=round(rng.uniform(5.0, 20.0), 2), vel=0.0)
    case = dict(kind=kind, eps=round(math.exp(rng.uniform(math.log(1e-3), math.log(0.1))), 5),
                dt=round(math.exp(rng.uniform(math.log(1e-3), math.log(2e-2))), 5), V=round(rng.uniform(1.0, 30.0), 2),
                vel=rng.choice([0.0, 0.1, 0.5]))
    family = rng.choice(["uniform", "band", "band", "random", "uniform2", "random2"])
    if family == "uniform":
        case.update(mesh="uniform", dim=3, level=rng.randint(3, 7), periodic=rng.choice([0, 0, 3]))
    elif family == "band":
        lv = rng.randint(2, 5)
        case.update(mesh="band", dim=3, level=lv, fine=lv + rng.randint(1, 3), band=round(rng.uniform(0.01, 0.2), 4))
    elif family == "random":
        case.update(mesh="random", dim=3, level=rng.randint(1, 2), fine=4, frac=round(rng.uniform(0.1, 0.4), 3),
                    tree=rng.randint(0, 999), periodic=rng.choice([0, 1]))
    elif family == "uniform2":
        case.update(mesh="uniform", dim=2, level=rng.randint(4, 9))
    else:
        case.update(mesh="random", dim=2, level=rng.randint(2, 3), fine=rng.randint(5, 6),
                    frac=round(rng.uniform(0.1, 0.4), 3), tree=rng.randint(0, 999), periodic=rng.choice([0, 1]))
    return case


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=2)
def _mesh(kind, dim, level, fine, band, frac, tree, periodic):
    """A program keeps one mesh for all the states and steps on it."""
    if kind == "uniform":
        oc = W.uniform_octants(dim, level)
    elif kind == "band":
        oc = W.membrane_band_octants(level, fine, band)
    else:
        oc = W.random_balanced_octants(dim, level, fine, frac, tree, periodic)
    return pnp.Mesh(W.with_periodic(oc, periodic))


def mesh_of(case):
    return _mesh(case["mesh"], case["dim"], case["level"], case.get("fine", 0), case.get("band", 0.0),
                 case.get("frac", 0.0), case.get("tree", 0), case.get("periodic", 0))


class Inputs:
    """Seeded device fields: smooth perturbations of a charged layer at the membrane under a
    linear potential, with the nodal noise of the runs' initial states."""

    def __init__(self, case, mesh, seed):
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed))
        self.g, self.dim, self.n = g, mesh.dim, mesh.n_nodes
        self.x = torch.from_numpy(mesh.ijk.astype(np.float64)).to(DEV) / 2.0**mesh.max_level
        self.V, self.lam, self.vel = case["V"], max(case["eps"], 0.02), case["vel"]

    def rand(self, *shape):
        return 2.0 * torch.rand(*shape, generator=self.g, device=DEV, dtype=F64) - 1.0

    def modes(self, m=4):
        k = torch.randint(1, 4, (m, self.dim), generator=self.g, device=DEV).to(F64)
        return torch.sin(2 * math.pi * (self.x @ k.T) + math.pi * self.rand(m)) @ self.rand(m) / m

    def state(self):
        z = self.x[:, -1]
        layer = torch.exp(-z / self.lam)
        U = torch.empty(self.n, 3, dtype=F64, device=DEV)
        U[:, 0] = 1.0 + layer + 0.1 * self.modes() + 1e-3 * self.rand(self.n)
        U[:, 1] = 1.0 - 0.5 * layer + 0.1 * self.modes() + 1e-3 * self.rand(self.n)
        U[:, 2] = self.V * z + 0.2 * self.modes() + 1e-3 * self.rand(self.n)
        return U

    def initial(self):
        """The start of a run: neutral with noise 1e-3, linear potential."""
        U = torch.empty(self.n, 3, dtype=F64, device=DEV)
        U[:, :2] = 1.0 + 1e-3 * self.rand(self.n, 2)
        U[:, 2] = self.V * self.x[:, -1]
        return U

    def direction(self):
        d = self.rand(self.n, 3)
        return d / d.norm()

    def velocity(self, m=6):
        """Divergence-free Fourier sums (amplitudes orthogonal to the wave vectors)."""
        if self.vel == 0.0:
            return torch.zeros(self.n, self.dim, dtype=F64, device=DEV)
        k = torch.randint(1, 4, (m, self.dim), generator=self.g, device=DEV).to(F64)
        a = self.rand(m, self.dim)
        a = a - (a * k).sum(1, keepdim=True) / (k * k).sum(1, keepdim=True) * k
        v = torch.sin(2 * math.pi * (self.x @ k.T) + math.pi * self.rand(m)) @ a
        return (self.vel / v.square().sum(1).mean().sqrt()) * v


def _params(case):
    kw = dict(eps=case["eps"], dt=case["dt"], **BDF2)
    if case["kind"] in ("time_step", "coupled_step"):
        kw["newton_rtol"] = NEWTON_RTOL
        if case["precision"] == "mixed":
            kw.update(MIXED_KW)
    if case["kind"] == "coupled_step":
        kw.update(NS_KW)
    return pnp.default_params(**kw)


def _bcs(case):
    return W.membrane_bcs(case["dim"], case["V"], 2.0)


def _mlp_weights(seed):
    r = np.random.default_rng(seed)
    sizes = [(K0, HID), (HID, HID), (HID, HID), (HID, NOUT)]
    return [(r.standard_normal(s).astype(np.float32) * math.sqrt(2.0 / s[0]),
             (0.1 * r.standard_normal(s[1])).astype(np.float32)) for s in sizes]


def _pack(ws):
    return np.concatenate([np.concatenate([w.reshape(-1), b]) for w, b in ws]).astype(np.float32)


def _mlp_inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    X = torch.randn(case["rows"], K0, generator=g, device=DEV)
    Y = torch.randn(case["rows"], NOUT, generator=g, device=DEV)
    return X, Y


def _fields(case, mesh, seed):
    """Every device input of a case, in a fixed order of generation."""
    I = Inputs(case, mesh, seed)
    f = {}
    if case["kind"] in ("time_step", "coupled_step"):
        f["U"] = I.initial()
        f["Uk"] = f["U"]
        f["Ukm1"] = I.initial()
        f["vk"] = f["vkm1"] = I.velocity()
        return f
    f["U"], f["Uk"], f["Ukm1"] = I.state(), I.state(), I.state()
    f["vk"], f["vkm1"] = I.velocity(), I.velocity()
    if case["kind"].startswith("jv"):
        f["D"] = I.direction()
    if case["kind"].startswith("ns"):
        f["X"] = I.rand(I.n, 4)
    return f


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind.startswith("mlp"):
        mesh = _mesh("uniform", 3, 2, 0, 0.0, 0.0, 0, 0)
        ctx = pnp.Context(mesh, pnp.default_params(), stream)
        ctx.mlp_init(0)
        ctx.mlp_set_weights(_pack(_mlp_weights(seed)))
        X, Y = _mlp_inputs(case, seed)
        out = torch.empty(case["rows"], NOUT, device=DEV)
        grad = torch.empty(pnp.PNP_MLP_PARAMS, device=DEV)
        return dict(case=case, ctx=ctx, X=X, Y=Y, out=out, grad=grad)
    mesh = mesh_of(case)
    ctx = pnp.Context(mesh, _params(case), stream)
    ctx.set_bcs(_bcs(case))
    f = _fields(case, mesh, seed)
    s = dict(case=case, ctx=ctx, mesh=mesh, **f)
    if kind in ("time_step", "coupled_step"):
        if kind == "coupled_step":
            ctx.ns_set_bcs(*_no_slip(case["dim"]))
        ctx.set_field(pnp.PNP_FIELD_U, f["U"])  # a run's states meet the boundary and hanging constraints
        ctx.make_consistent()
        s["Uk"] = torch.empty_like(f["U"])
        ctx.get_field(pnp.PNP_FIELD_U, s["Uk"])
        ctx.set_field(pnp.PNP_FIELD_U, f["Ukm1"])
        ctx.make_consistent()
        s["Ukm1"] = torch.empty_like(f["U"])
        ctx.get_field(pnp.PNP_FIELD_U, s["Ukm1"])
        s["out"] = torch.empty_like(f["U"])
        s["vel"] = torch.empty_like(f["vk"])
        s["ns0"] = torch.zeros(mesh.n_nodes, 4, dtype=F64, device=DEV)
        s["ns"] = torch.empty_like(s["ns0"])
        return s
    ctx.set_field(pnp.PNP_FIELD_U_PREV, f["Uk"])
    ctx.set_field(pnp.PNP_FIELD_U_PREV2, f["Ukm1"])
    if kind.startswith("ns"):
        ctx.ns_set_bcs(*_no_slip(case["dim"]))
        ctx.set_field(pnp.PNP_FIELD_VELOCITY, f["vk"])
        ctx.set_field(pnp.PNP_FIELD_VELOCITY_PREV, f["vkm1"])
        s["X"] = f["X"] if kind == "ns_matvec64" else f["X"].float()
        s["out"] = torch.empty_like(s["X"])
        return s
    ctx.set_field(pnp.PNP_FIELD_ADVECTION, f["vk"])
    if kind == "residual":
        s["out"] = torch.empty_like(f["U"])
    else:
        s["D"] = f["D"] if kind == "jv64" else f["D"].float()
        s["out"] = torch.empty_like(s["D"])
    if kind == "jv_linearized":
        ctx.linearize(f["U"])  # once per Krylov solve, for many directions
    return s


def _no_slip(dim):
    t = np.zeros((2 * dim, 4), np.int32)
    t[:, :3] = pnp.PNP_DIRICHLET
    return t, np.zeros((2 * dim, 4))


def run(s):
    kind, ctx = s["case"]["kind"], s["ctx"]
    if kind == "residual":
        return ctx.residual(s["U"], s["out"])
    if kind == "jv64":
        return ctx.jv(s["U"], s["D"], s["out"], pnp.PNP_F64)
    if kind == "jv32":
        return ctx.jv(s["U"], s["D"], s["out"], pnp.PNP_F32)
    if kind == "jv_linearized":
        return ctx.jv_linearized(s["D"], s["out"])
    if kind == "ns_matvec64":
        return ctx.ns_matvec(s["X"], s["out"], pnp.PNP_F64)
    if kind == "ns_matvec32":
        return ctx.ns_matvec(s["X"], s["out"], pnp.PNP_F32)
    if kind == "mlp_forward":
        return ctx.mlp_forward(s["X"], s["out"])
    if kind == "mlp_loss_grad":
        loss = ctx.mlp_loss_grad(s["X"], s["Y"], s["grad"])
        return {"grad": s["grad"], "loss": loss}
    # a step resumed from a stored history
    ctx.set_field(pnp.PNP_FIELD_U, s["Uk"])
    ctx.set_field(pnp.PNP_FIELD_U_PREV, s["Uk"])
    ctx.set_field(pnp.PNP_FIELD_U_PREV2, s["Ukm1"])
    ctx.set_field(pnp.PNP_FIELD_VELOCITY, s["vk"])
    ctx.set_field(pnp.PNP_FIELD_VELOCITY_PREV, s["vkm1"])
    ctx.set_step_count(1)
    if kind == "time_step":
        ctx.time_step()
        return ctx.get_field(pnp.PNP_FIELD_U, s["out"])
    ctx.set_field(pnp.PNP_FIELD_NS, s["ns0"])
    ctx.coupled_step()
    return {"U": ctx.get_field(pnp.PNP_FIELD_U, s["out"]), "velocity": ctx.get_field(pnp.PNP_FIELD_VELOCITY, s["vel"]),
            "ns": ctx.get_field(pnp.PNP_FIELD_NS, s["ns"])}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind.startswith("mlp"):
        B, P = case["rows"], pnp.PNP_MLP_PARAMS
        mm = 2.0 * (K0 * HID + 2 * HID * HID + HID * NOUT) * B
        if kind == "mlp_forward":
            return dict(bytes=4.0 * B * (K0 + NOUT) + 2.0 * P, flops=mm)
        # weight gradients cost the forward once more, activations' gradients all layers but the first
        return dict(bytes=4.0 * B * (K0 + NOUT) + 2.0 * P + 4.0 * P, flops=3 * mm - 2.0 * K0 * HID * B)
    m = mesh_of(case)
    N, E, d = float(m.n_nodes), float(m.n_elem), m.dim
    conn = E * (4.0 * 2**d + 1) + 17.0 * m.n_hanging
    q = 2.0**d  # Gauss points (and corners) of an element
    # values and gradients of a field at the points by 1D factors, the tests by their transposes
    interp, test = q * (3 * d + d * d), q * (3 * d + d * d)
    if kind == "residual":
        by, fl = 8.0 * N * (3 + 6 + d + 3), E * ((3 + 2 + d + 3) * interp + 40 * q)
    elif kind == "jv64":
        by, fl = 8.0 * N * (3 + 6 + d + 3 + 3), E * ((6 + 2 + d + 3) * interp + 80 * q)
    elif kind == "jv32":
        by, fl = 8.0 * N * (3 + 6 + d) + 4.0 * N * 6, E * ((6 + 2 + d + 3) * interp + 80 * q)
    elif kind == "jv_linearized":  # the state of the linearisation, the direction and the result
        by, fl = 4.0 * N * (3 + 2 + d + 3 + 3), E * ((6 + 2 + d + 3) * interp + 80 * q)
    elif kind == "ns_matvec64":
        by, fl = 8.0 * N * (4 + 2 * d + 4), E * ((d + 1) * (interp + test) + d * interp + 60 * q)
    elif kind == "ns_matvec32":
        by, fl = 4.0 * N * (4 + d + 4) + 16.0 * d * N, E * ((d + 1) * (interp + test) + d * interp + 60 * q)
    else:  # a step: its fields once, and one residual and one Jacobian action
        by, fl = 8.0 * N * (3 + 3 + 2 * d + 3), E * (2 * (3 + 2 + d + 3) * interp + 120 * q)
        if kind == "coupled_step":
            by, fl = by + 8.0 * N * (8 + d), fl + E * ((d + 1) * (interp + test) + 60 * q)
    return dict(bytes=by + conn, flops=fl)


# ------------------------------------------------------------------ the same in 64 bits
class Space:
    """Q1 space of a mesh in torch FP64: element corners as weighted independent nodes."""

    def __init__(self, mesh, periodic):
        d, L = mesh.dim, mesh.max_level
        self.d, self.n, self.size = d, mesh.n_nodes, 1 << L
        anchors, levels = mesh.elements()
        ijk = torch.from_numpy(mesh.ijk.astype(np.int64)).to(DEV)
        self.ijk, self.per = ijk, [bool(periodic >> k & 1) for k in range(d)]
        key, order = torch.sort(self._key(2 * ijk))
        a = torch.from_numpy(anchors.astype(np.int64)).to(DEV)
        s = torch.ones(len(levels), dtype=torch.int64, device=DEV) << (L - torch.from_numpy(levels.astype(np.int64)).to(DEV))
        self.h = s.to(F64) / self.size

        def find(p2):  # node at twice the coordinates, -1 where there is none
            k = self._key(p2)
            i = torch.searchsorted(key, k).clamp(max=self.n - 1)
            return torch.where(key[i] == k, order[i], torch.full_like(i, -1))

        bits = [torch.tensor([c >> k & 1 for k in range(d)], device=DEV) for c in range(1 << d)]
        conn = torch.stack([find(2 * (a + b * s[:, None])) for b in bits], 1)
        # a hanging node is the midpoint of an edge or the centre of a face of a coarser element
        self.hang = torch.from_numpy(mesh.hanging).to(DEV)
        par = torch.full((self.n, 4), -1, dtype=torch.int64, device=DEV)
        for t in np.ndindex(*([3] * d)):
            ones = [k for k in range(d) if t[k] == 1]
            if not 1 <= len(ones) < d:
                continue
            i = find(2 * a + torch.tensor(t, device=DEV) * s[:, None])
            sel = (i >= 0) & self.hang[i.clamp(min=0)]
            corners = [c for c in range(1 << d) if all((c >> k & 1) == t[k] // 2 for k in range(d) if t[k] != 1)]
            for j, c in enumerate(corners):
                par[i[sel], j] = conn[sel, c]
        self.par = torch.where(par >= 0, par, torch.zeros_like(par))
        self.wpar = (par >= 0).to(F64) / (par >= 0).sum(1, keepdim=True).clamp(min=1)
        self.conn = conn
        g = 1.0 / math.sqrt(3.0)
        sg = torch.tensor([[1.0 if c >> k & 1 else -1.0 for k in range(d)] for c in range(1 << d)], dtype=F64, device=DEV)
        f = 0.5 * (1.0 + sg[None] * (g * sg)[:, None])  # [point][corner][axis]
        self.N = f.prod(2)
        self.dN = torch.stack([0.5 * sg[None, :, k] * torch.cat([f[:, :, :k], f[:, :, k + 1:]], 2).prod(2)
                               for k in range(d)], 2) * 2.0  # times 1 / h

    def _key(self, p2):
        base, k = 2 * self.size + 1, torch.zeros(p2.shape[0], dtype=torch.int64, device=DEV)
        for x in range(self.d):
            c = p2[:, x] % (2 * self.size) if self.per[x] else p2[:, x]
            k = k * base + c
        return k

    def extend(self, u):
        """Nodal values with the hanging nodes interpolated."""
        return torch.where(self.hang[:, None], torch.einsum("np,npf->nf", self.wpar, u[self.par]), u)

    def at_points(self, u, e0, e1):
        """Values [e][q][f] and gradients [e][q][f][k] of extended nodal values."""
        uc = u[self.conn[e0:e1]]
        return torch.einsum("qc,ecf->eqf", self.N, uc), torch.einsum("qck,ecf->eqfk", self.dN, uc) / self.h[e0:e1, None, None, None]

    def tested(self, out, S, Phi, e0, e1):
        h = self.h[e0:e1]
        r = torch.einsum("qc,eqf->ecf", self.N, S) + torch.einsum("qck,eqfk->ecf", self.dN, Phi) / h[:, None, None]
        r = r * ((0.5 * h) ** self.d)[:, None, None]
        return out.index_add(0, self.conn[e0:e1].reshape(-1), r.reshape(-1, r.shape[2]))

    def rows(self, out, u, types, values):
        """Hanging contributions to the parents, then constraint and Dirichlet rows."""
        hr = torch.where(self.hang[:, None], out, torch.zeros_like(out))
        out = out - hr
        for p in range(4):
            out = out.index_add(0, self.par[:, p], self.wpar[:, p, None] * hr)
        out = torch.where(self.hang[:, None], u - self.extend(u), out)
        for face in range(2 * self.d):
            k = face // 2
            if self.per[k]:
                continue
            on = (self.ijk[:, k] == (self.size if face & 1 else 0)) & ~self.hang
            for f in range(out.shape[1]):
                if types[face][f] == pnp.PNP_DIRICHLET:
                    row = on[:, None] & (torch.arange(out.shape[1], device=DEV) == f)
                    out = torch.where(row, u - float(values[face][f]), out)
        return out

    def chunks(self, step=1 << 18):
        E = self.conn.shape[0]
        return [(e, min(E, e + step)) for e in range(0, E, step)]


def _tau(sp, case, vv, e0, e1, c2=1.0):
    G = (2.0 / sp.h[e0:e1, None]) ** 2
    return (4.0 / case["dt"] ** 2 + G * vv + 6.0 * c2 * sp.d * G * G) ** -0.5


def _residual(sp, case, U, Uk, Ukm1, vel):
    b0, b1, b2 = (BDF2[k] / case["dt"] for k in ("beta0", "beta1", "beta2"))
    bcs = _bcs(case)
    X = [sp.extend(u) for u in (U, Uk, Ukm1, vel)]
    out = torch.zeros_like(U)
    for e0, e1 in sp.chunks():
        u, g = sp.at_points(X[0], e0, e1)
        hist = b1 * sp.at_points(X[1], e0, e1)[0] + b2 * sp.at_points(X[2], e0, e1)[0]
        v = sp.at_points(X[3], e0, e1)[0]
        tau = _tau(sp, case, (v * v).sum(2), e0, e1)
        S, Phi, tR = [], [], []
        for f, z in ((0, 1.0), (1, -1.0)):
            dt_c = b0 * u[..., f] + hist[..., f]
            P = v - z * g[:, :, 2]
            tR.append(tau * (dt_c + (P * g[:, :, f]).sum(2)))
            S.append(dt_c + (v * g[:, :, f]).sum(2))
            Phi.append(g[:, :, f] + z * u[..., f, None] * g[:, :, 2] + tR[f][..., None] * P)
        S.append(u[..., 1] - u[..., 0] + tR[0] - tR[1])
        Phi.append(2.0 * case["eps"] ** 2 * g[:, :, 2])
        out = sp.tested(out, torch.stack(S, 2), torch.stack(Phi, 2), e0, e1)
    return sp.rows(out, U, bcs.types, bcs.values)


def _ns_matrix(sp, case, X, va):
    """A X of the NS rows with Sc = 1, no-slip walls and the pinned pressure."""
    d, b0 = sp.d, BDF2["beta0"] / case["dt"]
    Xe, ve = sp.extend(X), sp.extend(va)
    out = torch.zeros_like(X)
    for e0, e1 in sp.chunks():
        x, g = sp.at_points(Xe, e0, e1)
        v = sp.at_points(ve, e0, e1)[0]
        tau = _tau(sp, case, (v * v).sum(2), e0, e1)
        tsol = 1.0 / (d * (2.0 / sp.h[e0:e1, None]) ** 2 * tau)
        div = sum(g[:, :, i, i] for i in range(d))
        S, Phi, R = [], [], []
        for i in range(d):
            R.append(b0 * x[..., i] + (v * g[:, :, i]).sum(2) + g[:, :, 3, i])
            p = g[:, :, i] + (tau * R[i])[..., None] * v
            p = p + torch.nn.functional.one_hot(torch.tensor(i, device=DEV), d).to(F64) * (tsol * div)[..., None]
            S.append(R[i])
            Phi.append(p)
        for i in range(d, 3):
            S.append(torch.zeros_like(div))
            Phi.append(torch.zeros_like(g[:, :, 0]))
        S.append(div)
        Phi.append(tau[..., None] * torch.stack(R, 2))
        out = sp.tested(out, torch.stack(S, 2), torch.stack(Phi, 2), e0, e1)
    out = sp.rows(out, X, *_no_slip(d))
    pin = (sp.ijk == 0).all(1)
    out[pin, 3] = X[pin, 3]
    if d == 2:
        out[~sp.hang, 2] = X[~sp.hang, 2]
    return out


def _newton(sp, case, s0, Uk, Ukm1, vel):
    """The step's solution by Newton with dense Jacobians (columns by forward differentiation)."""
    n = 3 * sp.n
    U = s0.clone()
    F = lambda u: _residual(sp, case, u.reshape(-1, 3), Uk, Ukm1, vel).reshape(-1)  # noqa: E731
    for _ in range(30):
        r = F(U.reshape(-1))
        jv = lambda w: torch.func.jvp(F, (U.reshape(-1),), (w,))[1]  # noqa: E731
        J = torch.cat([torch.func.vmap(jv)(torch.eye(n, dtype=F64, device=DEV)[i:i + 256]) for i in range(0, n, 256)]).T
        d = torch.linalg.solve(J, -r)
        U = U + d.reshape(-1, 3)
        if d.norm() <= 1e-13 * U.norm():
            break
    return U


def _bf16(x):
    return x.bfloat16().to(F64)


def _network(ws, X):
    a = X
    for i, (w, b) in enumerate(ws):
        a = a @ w + b
        if i < 3:
            a = torch.nn.functional.gelu(a)
    return a


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("mlp"):
        # weights and inputs as the network takes them (BF16), everything after in 64 bits
        X, Y = _mlp_inputs(case, seed)
        ws = [(_bf16(torch.from_numpy(w).to(DEV)).requires_grad_(True), torch.from_numpy(b).to(DEV, F64).requires_grad_(True))
              for w, b in _mlp_weights(seed)]
        out = _network(ws, _bf16(X))
        if kind == "mlp_forward":
            return out.detach()
        loss = (out - Y.to(F64)).square().mean()
        grads = torch.autograd.grad(loss, [p for wb in ws for p in wb])
        return {"grad": torch.cat([g.reshape(-1) for g in grads]), "loss": float(loss.detach())}
    mesh = mesh_of(case)
    if kind in ("time_step", "coupled_step"):
        if kind == "coupled_step" or 3 * mesh.n_nodes > 4000:
            return None  # a nonlinear system too large for a dense solver
        s = prepare(case, seed)
        return _newton(Space(mesh, case.get("periodic", 0)), case, s["Uk"], s["Uk"], s["Ukm1"], s["vk"])
    f = _fields(case, mesh, seed)
    sp = Space(mesh, case.get("periodic", 0))
    if kind.startswith("ns"):
        X = f["X"] if kind == "ns_matvec64" else f["X"].float().to(F64)
        return _ns_matrix(sp, case, X, 2.0 * f["vk"] - f["vkm1"])
    F = lambda u: _residual(sp, case, u, f["Uk"], f["Ukm1"], f["vk"])  # noqa: E731
    if kind == "residual":
        return F(f["U"])
    D = f["D"] if kind == "jv64" else f["D"].float().to(F64)
    return torch.func.jvp(F, (f["U"],), (D,))[1]
