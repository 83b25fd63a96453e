"""Measured workloads of the library: what a user of the coupled fluid / rigid-body march has it do.

A case is one call sequence through the public entry points (``Solver``, ``objective``): the gradient
of one design (forward march, reverse sweep, sensitivity), the objective alone, the paper-form adjoint,
or the design chain with its volume constraint. The problems are those of ``workloads.config`` and
``workloads.verification`` and the benchmark's fluid grids, with the march cut to a few checkpoint
segments so that a pass stays short; ``draw`` varies grid, body, motion, boundary kinds, precision and
checkpointing over the same ranges. A handle with FP32 fields gives FP32 results (the design is then an
FP32 parameter, the state is FP32); a handle with FP64 fields gives FP64 results.

``exact`` is a plain torch FP64 statement of the same method, differentiated by autograd.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as TF
from torch.utils.checkpoint import checkpoint

from paper_2601_18272_gb300.autograd import objective
from paper_2601_18272_gb300.lks import Solver
from workloads import (BC_INFLOW_OUTFLOW, BC_PERIODIC, BC_PRESSURE, BC_WALL, CKPT_BF16, CKPT_BINOMIAL, CKPT_FP16,
                       CKPT_FP32, CKPT_STORE_ALL, CKPT_UNIFORM, DOF_ROT, DOF_TX, DOF_TY, DOF_TZ, ROT_FREE,
                       W_BILINEAR, W_COS4, Problem, inertia_tensor, mass_properties)
from workloads.synth import design_offsets

DEVICE = "cuda"


def _case(**kw):
    """A case with the defaults of the 2D rotating-body workload filled in."""
    c = dict(action="gradient", dim=2, nx=512, ny=256, nz=1, nd=128, body="solid", motion="rot", flow="inflow",
             weight="cos", bits=32, steps=200, itr=5, ckpt="uniform", every=100, fmt="native", re=200.0,
             filter=0.0, beta=0.0, cyclic=1)
    c.update(kw)
    return c


def listed():
    return [
        # the design chain and volume constraint of one optimisation iterate, without a march: the
        # smallest call a user makes, latency only (256^2 turbine design, filter, projection, cyclic)
        _case(name="design_chain_256", action="constraint", nx=1024, ny=512, nd=256, steps=1, every=1, filter=3.0,
              beta=4.0, cyclic=4),
        # the paper's small 2D sail in FP64, every state stored, at its full length: the case a user
        # checks derivatives on
        _case(name="sail_80x40_fp64", nx=80, ny=40, nd=16, motion="x", weight="linear", bits=64, steps=400,
              ckpt="all", every=0, re=100.0),
        # Appendix B's pressure-driven channel between walls, rotating body, FP64
        _case(name="channel_600x100_fp64", nx=600, ny=100, nd=20, flow="channel", bits=64, steps=200, ckpt="all",
              every=0),
        # the benchmark workload: 2D turbine, FP32 fields, two checkpoint segments
        _case(name="turbine_512x256"),
        # the same march without its gradient: an objective evaluation (line search, finite differences)
        _case(name="turbine_512x256_forward", action="forward", steps=300),
        # the same body with the paper's own adjoint
        _case(name="turbine_512x256_paper", action="paper", steps=100, every=50),
        # 2D body free in x, y and angle, BF16 checkpoints: the larger 2D design
        _case(name="sailturbine_1024x512", nx=1024, ny=512, nd=256, motion="xyrot", steps=100, every=50, fmt="bf16",
              re=500.0),
        # a large 2D channel around a body: full-grid kernels beyond L2, through the autograd form
        _case(name="open_2d_4096x2048", action="autograd", nx=4096, ny=2048, nd=64, steps=20, every=10, re=100.0),
        # 3D body translating in x, y, z
        _case(name="body3d_128x64x64", dim=3, nx=128, ny=64, nz=64, nd=48, motion="xyz", steps=40, every=20,
              re=100.0),
        # 3D body in a duct with walls on an odd, ragged grid, turning about one axis
        _case(name="duct3d_157x67x70", dim=3, nx=157, ny=67, nz=70, nd=31, motion="rot", flow="duct", steps=24,
              every=12, re=100.0),
        # six-DOF 3D turbine (ball domain) with binomial BF16 snapshots
        _case(name="turbine3d_6dof", dim=3, nx=256, ny=128, nz=128, nd=96, body="ball", motion="free",
              flow="periodic", steps=12, ckpt="binomial", every=4, fmt="bf16", re=300.0),
        # the largest grid: a small 3D body in 33.5 million cells
        _case(name="open_3d_512x256x256", dim=3, nx=512, ny=256, nz=256, nd=24, motion="xyz", steps=6, every=3,
              re=100.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _design_edge(rng, cells, share):
    """A design edge whose rotated support box fits `share` of the given extent (diagonal included)."""
    top = int((share * cells - 14) / (1.7321 if share < 0.9 else 1.4143))
    return max(4, min(top, int(_log(rng, 6, max(7, top)))))


def draw(rng):
    kind = rng.choice(["chain", "small64", "channel", "mid2d", "forward", "paper", "big2d", "body3d", "duct3d",
                       "free3d", "big3d"])
    itr = rng.choice([1, 3, 4, 5, 5, 5, 6])
    if kind == "chain":
        nd = int(_log(rng, 20, 300))
        return _case(action="constraint", nx=4 * nd + 64, ny=2 * nd + 32, nd=nd, steps=1, every=1,
                     filter=rng.choice([0.0, 1.5, 2.0, 3.0, 4.5]), beta=rng.choice([0.0, 2.0, 8.0]),
                     cyclic=rng.choice([1, 2, 4]))
    if kind in ("small64", "channel"):
        ny = int(_log(rng, 36, 130))
        nx = int(ny * rng.uniform(2.0, 5.0))
        return _case(nx=nx, ny=ny, nd=_design_edge(rng, ny, 0.95), motion=rng.choice(["x", "xyrot", "rot"]),
                     flow="inflow" if kind == "small64" else "channel", weight=rng.choice(["cos", "linear"]),
                     bits=64, steps=rng.randint(40, 300), itr=itr, ckpt="all", every=0, re=rng.uniform(40, 200))
    if kind in ("mid2d", "forward", "paper"):
        ny = int(_log(rng, 96, 640))
        nx = int(ny * rng.uniform(1.8, 3.0))
        every = rng.choice([20, 37, 50, 64])
        return _case(action={"mid2d": rng.choice(["gradient", "autograd"]), "forward": "forward", "paper": "paper"}[kind],
                     nx=nx, ny=ny, nd=_design_edge(rng, ny, 0.95), motion=rng.choice(["x", "xyrot", "rot"]),
                     steps=rng.randint(30, 140), itr=itr, every=every, fmt=rng.choice(["native", "bf16", "fp16"]),
                     re=rng.uniform(60, 500), weight=rng.choice(["cos", "cos", "linear"]))
    if kind == "big2d":
        ny = int(_log(rng, 1000, 2400))
        nx = int(ny * rng.uniform(1.3, 2.2))
        return _case(nx=nx, ny=ny, nd=rng.randint(16, 300), motion=rng.choice(["xyrot", "rot"]), itr=itr,
                     flow=rng.choice(["inflow", "periodic"]), steps=rng.randint(8, 16), every=rng.randint(4, 8),
                     re=rng.uniform(100, 500))
    if kind in ("body3d", "duct3d"):
        ny, nz = int(_log(rng, 40, 110)), int(_log(rng, 40, 110))
        nx = int(max(ny, nz, 64) * rng.uniform(1.6, 2.4))
        if kind == "body3d":
            nx -= nx % 4
        else:  # a grid the walled 3D form takes: its last column and row hold more than one cell
            nx += int(nx % 32 == 1)
            ny += int(ny % 16 == 1)
        return _case(dim=3, nx=nx, ny=ny, nz=nz, nd=_design_edge(rng, min(ny, nz), 0.95),
                     motion=rng.choice(["xyz", "xyzrot", "rot"]), itr=itr,
                     flow="inflow" if kind == "body3d" else "duct", steps=rng.randint(6, 24), every=rng.randint(4, 12),
                     re=rng.uniform(40, 150))
    if kind == "free3d":
        ny = 4 * rng.randint(12, 30)
        return _case(dim=3, nx=2 * ny, ny=ny, nz=ny, nd=_design_edge(rng, ny, 0.85), body=rng.choice(["ball", "solid"]),
                     motion="free", flow="periodic", steps=rng.randint(5, 12), itr=itr, ckpt="binomial",
                     every=rng.randint(2, 5), fmt=rng.choice(["native", "bf16"]), re=rng.uniform(100, 300))
    ny, nz = rng.randint(128, 240), rng.randint(128, 240)
    return _case(dim=3, nx=4 * rng.randint(40, 120), ny=ny, nz=nz, nd=rng.randint(10, 30), itr=itr,
                 motion=rng.choice(["xyz", "rot"]), steps=rng.randint(3, 6), every=rng.randint(2, 4),
                 re=rng.uniform(60, 150))


# ---- the problem a case states ------------------------------------------------------------------

_MOTION = {"x": DOF_TX, "rot": DOF_ROT, "xyrot": DOF_TX | DOF_TY | DOF_ROT, "xyz": DOF_TX | DOF_TY | DOF_TZ,
           "xyzrot": DOF_TX | DOF_TY | DOF_TZ | DOF_ROT, "free": DOF_TX | DOF_TY | DOF_TZ | DOF_ROT}
_FLOW = {"inflow": (BC_INFLOW_OUTFLOW, BC_PERIODIC, BC_PERIODIC), "periodic": (BC_PERIODIC,) * 3,
         "channel": (BC_PRESSURE, BC_WALL, BC_PERIODIC), "duct": (BC_INFLOW_OUTFLOW, BC_WALL, BC_WALL)}


def _design(c, seed):
    """gamma in [0, 1], x fastest: smoothed uniform noise (2D) or a refined coarse lattice (3D)."""
    gen = torch.Generator().manual_seed(int(seed))
    nd = c["nd"]
    if c["dim"] == 2:
        g = torch.rand((1, 1, nd, nd), generator=gen, dtype=torch.float64)
        for _ in range(2):
            g = TF.avg_pool2d(g, 3, 1, 1, count_include_pad=False)
        # heavier on one side of the pivot, as a design under way is: a stream then turns the body, where
        # on plain noise the torque would be a difference of large sums
        side = (torch.arange(nd, dtype=torch.float64) - (nd - 1) / 2.0) * (8.0 / nd)
        g = g * (0.2 + 0.8 * torch.sigmoid(side))[None, None, :, None]
    else:
        m = -(-nd // 8) + 1
        g = TF.interpolate(torch.rand((1, 1, m, m, m), generator=gen, dtype=torch.float64), size=(nd,) * 3,
                           mode="trilinear", align_corners=True)
    g = g.reshape(-1)
    if c["body"] == "ball":
        r = torch.from_numpy(design_offsets((nd, nd, nd), 3))
        g = g * ((r ** 2).sum(1) <= (nd / 2.0 - 2.0) ** 2)
    if c["bits"] == 32:  # an FP32 design parameter
        g = g.float().double()
    return g


def _problem(c, seed):
    """(Problem, gamma) of a case; mass and inertia follow the design as in the workloads."""
    g = _design(c, seed)
    dim, nd = c["dim"], c["nd"]
    free = c["motion"] == "free"
    size = (nd, nd, nd if dim == 3 else 1)
    mass, inertia = mass_properties(g.numpy(), size, dim, 2)
    tensor = inertia_tensor(g.numpy(), size) if free else (0.0,) * 9
    w = [0.0] * (21 if free else 8)
    w[6 if "rot" in c["motion"] or free else 0] = 1.0
    channel = c["flow"] == "channel"
    centre = (c["nx"] * (0.375 if free else 0.25 if c["nx"] >= 2 * c["ny"] else 0.375) + (0.3 if dim == 3 else 0.0),
              c["ny"] / 2.0, c["nz"] / 2.0 if dim == 3 else 0.0)
    half = math.ceil((1.0 if _MOTION[c["motion"]] & DOF_ROT == 0 else 1.7321 if free else 1.4143) * nd / 2) + 8  # the body starts clear of the open planes
    if c["flow"] != "periodic":
        centre = (max(centre[0], float(min(half, c["nx"] // 2))),) + centre[1:]
    P = Problem(dim=dim, nx=c["nx"], ny=c["ny"], nz=c["nz"], ndx=nd, ndy=nd, ndz=nd if dim == 3 else 1,
                body_centre=centre, rot_axis=ROT_FREE if free else 2, dof_mask=_MOTION[c["motion"]], mass=mass,
                inertia=inertia, nu=0.1 if channel else 0.05 * nd / c["re"], u_in=0.0 if channel else 0.05,
                dp=1e-2 if channel else 0.0, bc=_FLOW[c["flow"]], kappa_max=200.0 if channel else 1.0,
                q=1e-2 if channel else 0.1, weight_kind=W_COS4 if c["weight"] == "cos" else W_BILINEAR,
                n_steps=c["steps"], n_itr=c["itr"], obj_weights=tuple(w), field_precision=c["bits"],
                ckpt_policy={"all": CKPT_STORE_ALL, "uniform": CKPT_UNIFORM, "binomial": CKPT_BINOMIAL}[c["ckpt"]],
                ckpt_every=c["every"], ckpt_format={"native": CKPT_FP32, "bf16": CKPT_BF16, "fp16": CKPT_FP16}[c["fmt"]],
                inertia_tensor=tensor, design_radius=nd / 2.0 - 2.0 if c["body"] == "ball" else 0.0,
                filter_radius=c["filter"], proj_beta=c["beta"], cyclic_order=c["cyclic"], name="case")
    return P, g


def _initial(P):
    """(p, u) a march starts from: the default impulsive stream, or in the pressure-driven channel a
    linear pressure drop with a parabolic profile (there the default, rest, would stay at rest until
    the pressure wave arrives). The body starts at rest."""
    if P.bc[0] != BC_PRESSURE:
        return None
    y = np.arange(P.ny) / (P.ny - 1.0)
    p = np.tile(P.dp * (1.0 - np.arange(P.nx) / (P.nx - 1.0)), P.ny)
    u = np.zeros((P.dim, P.n_cells))
    u[0] = np.repeat(0.2 * y * (1.0 - y), P.nx)
    return p, u


# ---- the calls ----------------------------------------------------------------------------------

def prepare(case, seed):
    """The handle (created once per problem by a user's program) and the design on the device."""
    P, g = _problem(case, seed)
    S = Solver(P)
    flow = _initial(P)
    if flow:
        S.set_initial_state(*flow)
    gamma = g.to(DEVICE)
    state = {"case": case, "solver": S, "gamma": gamma, "out": torch.empty_like(gamma),
             "type": torch.float32 if case["bits"] == 32 else torch.float64}
    if case["action"] == "autograd":
        state["parameter"] = gamma.to(state["type"]).requires_grad_(True)
    return state


def run(state):
    S, gamma, out, action = state["solver"], state["gamma"], state["out"], state["case"]["action"]
    np_type = np.float32 if state["case"]["bits"] == 32 else np.float64
    if action == "constraint":
        G = S.constraint(gamma, out)
        return {"G": np.float64(G), "dG": out}
    if action == "forward":
        J = S.forward(gamma)
        p, u = S.state()
        return {"J": np_type(J), "dofs": S.dof_history().astype(np_type), "p": p.astype(np_type), "u": u.astype(np_type)}
    if action == "autograd":
        x = state["parameter"]
        x.grad = None
        J = objective(x, S)
        J.backward()
        return {"J": J.detach().to(state["type"]), "dJ": x.grad}
    J = S.forward(gamma)
    if action == "paper":
        S.adjoint_alks(1.0)
    else:
        S.adjoint(1.0)
    S.sensitivity(out)
    return {"J": np_type(J), "dJ": out.to(state["type"])}


def work(case):
    """Bytes: the design in and the results out, and per time step the state read and written once
    (and in the reverse step the adjoint read and written and the velocity read). Floating-point
    operations: the predictor and its transpose per cell, the spread per design point and iteration."""
    dim, nd = case["dim"], case["nd"]
    esz = case["bits"] // 8
    N, ND = case["nx"] * case["ny"] * case["nz"], nd ** dim
    if case["action"] == "constraint":
        disc = max(1.0, math.pi * case["filter"] ** 2)
        return {"bytes": 16.0 * ND, "flops": (6.0 * disc + 20.0) * ND}
    fluid = 160.0 if dim == 2 else 420.0
    reach = (4 if case["weight"] == "cos" else 2) ** dim
    fwd_b, fwd_f = 2.0 * (dim + 1) * esz * N, fluid * N + case["itr"] * reach * ND * (8.0 + 4 * dim)
    if case["action"] == "forward":
        return {"bytes": case["steps"] * fwd_b + 8.0 * ND + (dim + 1) * esz * N, "flops": case["steps"] * fwd_f}
    rev_b = (3.0 * dim + 2) * esz * N
    return {"bytes": case["steps"] * (fwd_b + rev_b) + 16.0 * ND, "flops": 3.0 * case["steps"] * fwd_f}


# ---- the same in plain torch, FP64 ----------------------------------------------------------------

_C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)] + [
    (sx, sy, sz) for sz in (1, -1) for sy in (1, -1) for sx in (1, -1)]


class _Plain:
    """The march of one problem on fields shaped [..., (nz,) ny, nx]; axis a of space is tensor axis -1 - a."""

    def __init__(self, P):
        self.P, self.d = P, P.dim
        self.A = 4.5 * (1.0 / 6.0 - P.nu)
        self.c = _C2 if P.dim == 2 else _C3
        w0, w1, w2 = (4 / 9, 1 / 9, 1 / 36) if P.dim == 2 else (2 / 9, 1 / 9, 1 / 72)
        self.w = [w0 if sum(map(abs, c)) == 0 else w1 if sum(map(abs, c)) == 1 else w2 for c in self.c]
        self.cn = sum(c[0] ** 2 for c in self.c)
        self.n = (P.nx, P.ny, P.nz)[:P.dim]
        self.shape = tuple(reversed(self.n))
        r = torch.from_numpy(design_offsets((P.ndx, P.ndy, P.ndz), P.dim)).to(DEVICE)
        dom = torch.ones(len(r), dtype=torch.bool, device=DEVICE)
        if P.design_radius > 0:
            dom = (r ** 2).sum(1) <= P.design_radius ** 2
        self.dom, self.r = dom, r[dom]
        self.free = P.rot_axis == ROT_FREE
        if self.free:
            J = torch.tensor(P.inertia_tensor, dtype=torch.float64).reshape(3, 3)
            self.Jinv = torch.linalg.inv(J).to(DEVICE)

    def chain(self, gamma):
        """Cyclic expansion, conic filter over the design domain, Heaviside projection (2D designs)."""
        P = self.P
        g = gamma
        if P.cyclic_order > 1:
            at = torch.arange(P.ndx * P.ndy, device=gamma.device).reshape(P.ndy, P.ndx)
            rep = at
            for k in range(1, 4):
                if P.cyclic_order == 4 or k == 2:
                    rep = torch.minimum(rep, torch.rot90(at, k))
            g = gamma[rep.reshape(-1)]
        if P.filter_radius > 0:
            R, m = P.filter_radius, int(P.filter_radius)
            e = torch.arange(-m, m + 1, dtype=torch.float64, device=gamma.device)
            k = torch.clamp((R - torch.sqrt(e[:, None] ** 2 + e[None, :] ** 2)) / R, min=0)
            image = g.reshape(P.ndy, P.ndx)
            pad = TF.pad(image, (m, m, m, m))
            ones = TF.pad(torch.ones_like(image), (m, m, m, m))
            a = w = 0
            for i in range(2 * m + 1):
                for j in range(2 * m + 1):
                    a = a + k[i, j] * pad[i:i + P.ndy, j:j + P.ndx]
                    w = w + k[i, j] * ones[i:i + P.ndy, j:j + P.ndx]
            g = (a / w).reshape(-1)
        if P.proj_beta > 0:
            b, eta = P.proj_beta, P.proj_eta
            g = (math.tanh(b * eta) + torch.tanh(b * (g - eta))) / (math.tanh(b * eta) + math.tanh(b * (1 - eta)))
        return g

    def _ghosts(self, u):
        """One ghost layer per axis: periodic wrap, copy of an open plane, odd reflection at a wall."""
        for a in range(self.d):
            ax, n, bc = u.dim() - 1 - a, self.n[a], self.P.bc[a]
            if bc == BC_PERIODIC:
                lo, hi = u.narrow(ax, n - 1, 1), u.narrow(ax, 0, 1)
            elif bc == BC_WALL:
                lo, hi = -u.narrow(ax, 1, 1), -u.narrow(ax, n - 2, 1)
            else:
                lo, hi = u.narrow(ax, 0, 1), u.narrow(ax, n - 1, 1)
            u = torch.cat([lo, u, hi], ax)
        return u

    def _at(self, padded, c):
        out = padded
        for a in range(self.d):
            out = out.narrow(out.dim() - 1 - a, 1 + c[a], self.n[a])
        return out

    def _gradient(self, ua):
        """d_b u_a, all b, of one velocity component."""
        g = self._ghosts(ua)
        return torch.stack([sum(c[b] * self._at(g, c) for c in self.c if c[b]) / self.cn for b in range(self.d)])

    def _moments(self, i, p, u, G, uu):
        c = self.c[i]
        cu = sum(c[a] * u[a] for a in range(self.d) if c[a])
        f = 3.0 * p - 1.5 * uu
        if any(c):
            quad = sum(c[a] * c[b] * G[a][b] for a in range(self.d) for b in range(self.d) if c[a] and c[b])
            f = f + 3.0 * cu + 4.5 * cu * cu + 2.0 * self.A * quad
        return torch.roll(self.w[i] * f, tuple(c[a] for a in range(self.d)), tuple(-1 - a for a in range(self.d)))

    def fluid(self, p, u):
        """Predictor and boundary values."""
        P, d = self.P, self.d
        big = p.numel() > 4_000_000
        call = (lambda f, *x: checkpoint(f, *x, use_reentrant=False)) if big else (lambda f, *x: f(*x))
        G = [call(self._gradient, u[a]) for a in range(d)]
        uu = (u * u).sum(0)
        ps, us = 0, [0] * d
        for i, c in enumerate(self.c):
            f = call(lambda *x, i=i: self._moments(i, x[0], x[1], x[2:2 + d], x[-1]), p, u, *G, uu)
            ps = ps + f
            us = [us[a] + c[a] * f if c[a] else us[a] for a in range(d)]
        ps = ps / 3.0
        s = torch.stack([ps] + us)
        for a in range(1, d):
            if P.bc[a] == BC_WALL:  # the wall rows of x-interior nodes; the x planes follow for every row
                ax, n = s.dim() - 1 - a, self.n[a]
                zero = torch.zeros_like(s.narrow(ax, 0, 1)[1:])
                s = torch.cat([torch.cat([s.narrow(ax, 1, 1)[:1], zero]), s.narrow(ax, 1, n - 2),
                               torch.cat([s.narrow(ax, n - 2, 1)[:1], zero])], ax)
        if P.bc[0] != BC_PERIODIC:
            n = self.n[0]
            first, last = s[..., 1:2], s[..., n - 2:n - 1]
            if P.bc[0] == BC_INFLOW_OUTFLOW:
                u_in = torch.zeros_like(first[1:])
                u_in[0] = P.u_in
                first = torch.cat([first[:1], u_in])
            else:
                first = torch.cat([torch.full_like(first[:1], P.dp), first[1:]])
            last = torch.cat([torch.zeros_like(last[:1]), last[1:]])
            s = torch.cat([first, s[..., 1:n - 1], last], -1)
        return s[0], s[1:]

    def _pose(self, s):
        """World offsets R r, the design points' solid velocity, and (R r) for the lever."""
        r = self.r
        if self.free:
            l = r @ s[12:21].reshape(3, 3).T
            return l, s[3:6] + torch.linalg.cross(s[9:12].expand_as(l), l)
        ct, st = torch.cos(s[6]), torch.sin(s[6])
        x, y = r[:, 0], r[:, 1]
        l = torch.stack([ct * x - st * y, st * x + ct * y, r[:, 2]], 1)
        turn = torch.stack([-l[:, 1], l[:, 0], torch.zeros_like(x)], 1)
        return l, s[3:6] + s[7] * turn

    def _spread(self, kappa, s):
        """Window indices [M, (2 half)^d], weights, lever, solid velocity under s."""
        P, d = self.P, self.d
        half = 2 if P.weight_kind == W_COS4 else 1
        l, us = self._pose(s)
        at, W, stride = 0, 1, 1
        for a in range(d):
            x = s[a] + l[:, a]
            cell = torch.floor(x.detach()).long()[:, None] + torch.arange(1 - half, half + 1, device=x.device)
            o = cell - x[:, None]
            if P.weight_kind == W_COS4:
                w = 0.25 * (1.0 + torch.cos(0.5 * math.pi * o))
            else:
                w = torch.where(o >= 0, 1.0 - o, 1.0 + o)
            w = torch.where(o.detach().abs() < half, w, torch.zeros_like(w))
            shape = [len(l)] + [1] * d
            shape[1 + a] = 2 * half
            at = at + (cell % self.n[a]).reshape(shape) * stride
            W = W * w.reshape(shape)
            stride *= self.n[a]
        return at.reshape(len(l), -1), W.reshape(len(l), -1), l, us

    def _brinkman(self, kappa, s, ustar, want_force):
        """u of the Brinkman update under s, or the force and torque it puts on the body."""
        d, N = self.d, ustar[0].numel()
        at, W, l, us = self._spread(kappa, s)
        put = lambda v: torch.zeros(N, dtype=W.dtype, device=W.device).index_add(0, at.reshape(-1), v.reshape(-1))  # noqa: E731
        kn = put(W * kappa[:, None])
        flat = ustar.reshape(d, -1)
        u = torch.stack([(flat[a] + kn * put(W * us[:, a:a + 1])) / (1.0 + kn) for a in range(d)])
        if not want_force:
            return u.reshape(ustar.shape)
        ref = torch.stack([(W * u[a][at]).sum(1) for a in range(d)], 1)
        f = kappa[:, None] * (ref - us[:, :d])
        if d == 2:
            f = torch.cat([f, torch.zeros_like(f[:, :1])], 1)
        return torch.cat([f.sum(0), torch.linalg.cross(l, f).sum(0)])

    def _eom(self, s, FT):
        P, mask = self.P, self.P.dof_mask
        free_axes = torch.tensor([1.0 if mask & (1 << a) else 0.0 for a in range(3)], dtype=s.dtype, device=s.device)
        u = s[3:6] + free_axes * FT[:3] / P.mass
        x = s[:3] + free_axes * u
        if not self.free:
            if not mask & DOF_ROT:
                return torch.cat([x, u, s[6:8]])
            om = s[7] + FT[5] / P.inertia
            return torch.cat([x, u, torch.stack([s[6] + om, om])])
        R = s[12:21].reshape(3, 3)
        h = s[6:9] + FT[3:]
        om = R @ (self.Jinv @ (R.T @ h))
        K = torch.stack([torch.zeros_like(om[0]), -om[2], om[1], om[2], torch.zeros_like(om[0]), -om[0], -om[1], om[0],
                         torch.zeros_like(om[0])]).reshape(3, 3)
        Q, term = torch.eye(3, dtype=s.dtype, device=s.device), torch.eye(3, dtype=s.dtype, device=s.device)
        for k in range(1, 14):  # exp([omega]x): one step turns by far less than one radian
            term = term @ K / k
            Q = Q + term
        return torch.cat([x, u, h, om, (Q @ R).reshape(-1)])

    def step(self, p, u, s, kappa):
        p, us = self.fluid(p, u)
        sk = s
        call = (lambda f, *x: checkpoint(f, *x, use_reentrant=False)) if len(kappa) > 50_000 else (lambda f, *x: f(*x))
        for k in range(self.P.n_itr):
            FT = call(lambda *x: self._brinkman(*x, True), kappa, sk, us)
            if k == self.P.n_itr - 1:
                u = call(lambda *x: self._brinkman(*x, False), kappa, sk, us)
            sk = self._eom(s, FT)
        return p, u, sk

    def start(self):
        P = self.P
        p = torch.zeros(self.shape, dtype=torch.float64, device=DEVICE)
        u = torch.zeros((self.d,) + self.shape, dtype=torch.float64, device=DEVICE)
        u[0] = P.u_in
        flow = _initial(P)
        if flow:
            p = torch.from_numpy(flow[0]).to(DEVICE).reshape(p.shape)
            u = torch.from_numpy(flow[1]).to(DEVICE).reshape(u.shape)
        s = torch.zeros(P.n_dof, dtype=torch.float64, device=DEVICE)
        s[:3] = torch.tensor(P.body_centre, dtype=torch.float64)
        if self.free:
            s[12:21] = torch.eye(3, dtype=torch.float64).reshape(-1)
        return p, u, s

    def kappa(self, gamma):
        P, gb = self.P, self.chain(gamma)
        return (P.kappa_max * P.q * gb / (1.0 - gb + P.q))[self.dom]


def _exact_cost(c):
    """Rough seconds of exact(): kernel launches and memory traffic of the plain march."""
    N, M = c["nx"] * c["ny"] * c["nz"], c["nd"] ** c["dim"] * (4 ** c["dim"] if c["weight"] == "cos" else 2 ** c["dim"])
    launches = (300 if c["dim"] == 2 else 900) + 120 * c["itr"]
    traffic = (N * (1500 if c["dim"] == 2 else 5000) + M * 500 * c["itr"]) * 8
    factor = 1 if c["action"] == "forward" else 4
    return c["steps"] * factor * (launches * 1e-5 + traffic / 4e12)


def exact(case, seed):
    P, g = _problem(case, seed)
    g = g.to(DEVICE)
    if case["action"] == "constraint":
        x = g.requires_grad_(True)
        plain = _Plain(P)
        G = plain.chain(x)[plain.dom].sum() / (P.v_min * int(plain.dom.sum())) - 1.0
        G.backward()
        return {"G": G.detach(), "dG": x.grad}
    if _exact_cost(case) > 18.0:
        return None
    plain = _Plain(P)
    states = [plain.start()]
    with torch.no_grad():
        kappa = plain.kappa(g)
        for _ in range(P.n_steps):
            states.append(plain.step(*states[-1], kappa))
            if case["action"] == "forward":
                states[-2] = (None, None, states[-2][2])
    w = torch.tensor(P.obj_weights, dtype=torch.float64, device=DEVICE)
    J = (w * states[-1][2]).sum()
    if case["action"] == "forward":
        p, u, _ = states[-1]
        return {"J": J, "dofs": torch.stack([x[2] for x in states]), "p": p.reshape(-1), "u": u.reshape(P.dim, -1)}
    if case["action"] == "paper":  # a discretised continuous adjoint: no plain derivative equals it
        return {"J": J, "dJ": None}
    x = g.requires_grad_(True)
    kappa = plain.kappa(x)
    leaf = kappa.detach().requires_grad_(True)
    lam = (torch.zeros_like(states[-1][0]), torch.zeros_like(states[-1][1]), w.clone())
    dk = torch.zeros_like(leaf)
    for t in range(P.n_steps, 0, -1):
        inputs = [v.detach().requires_grad_(True) for v in states[t - 1]]
        states[t] = None
        outs = plain.step(*inputs, leaf)
        pairs = [(o, l) for o, l in zip(outs, lam) if o.requires_grad]
        got = torch.autograd.grad([o for o, _ in pairs], inputs + [leaf], [l for _, l in pairs], allow_unused=True)
        lam = [torch.zeros_like(v) if q is None else q for v, q in zip(inputs, got[:3])]
        dk = dk + got[3]
    kappa.backward(dk)
    return {"J": J, "dJ": x.grad}
