"""Performance cases of the differentiable magneto-elastic MPM library.

What a user of this package has it do, at the sizes of the package's own
workloads (``paper_2503_22767_gb300.workloads``), tests and benchmark: rollouts
(forward only), design gradients (forward + checkpointed adjoint) in 2D and
3D, batches of candidates, solid boxes, a non-uniform field, one
allocation-free substep and the design maps with their optimiser step.
Everything is float32, the library's one data type.

    listed()            the fixed cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) inputs (from the seed alone) and the handle, on the GPU
    run(state)          one pass through the public entry points
    work(case)          bytes and operations one pass cannot do without
    exact(case, seed)   the same outputs from plain torch in 64 bits
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2503_22767_gb300 import binding as B
from paper_2503_22767_gb300 import workloads as W
from paper_2503_22767_gb300.design import PARAM_BOX, DesignMaps, adam_step
from paper_2503_22767_gb300.sim import MpmSim, Simulator

MU0 = 4.0e-7 * math.pi


def listed():
    return [
        # one substep of a small beam inside a caller's own latency-critical loop
        {"name": "substep_2d", "kind": "substep", "dim": 2, "res": 64, "per_axis": 2},
        # shape morphing of the 2D beam: one design gradient through autograd, every substep stored
        {"name": "beam_2d", "kind": "beam", "res": 64, "per_axis": 4, "steps": 200},
        # scoring a half-size 2D walker from host buffers (a candidate search without gradients)
        {"name": "rollout_2d", "kind": "rollout2", "scale": 0.5, "steps": 400, "every": 100},
        # the 2D locomotion body: one checkpointed design gradient
        {"name": "walker_2d", "kind": "walker2", "scale": 1.0, "steps": 400, "every": 100},
        # 64 uneven 2D walkers evaluated as one batch, with the options its tuning settles on
        {"name": "batch_2d", "kind": "batch2", "instances": 64, "n_lo": 5000, "n_hi": 40000, "steps": 100, "every": 50},
        # a 2D body held by a moving clamp above a frictional step (solid boxes)
        {"name": "clamp_2d", "kind": "clamp2", "scale": 0.6, "steps": 200, "every": 100},
        # three tasks of the 3D plate sharing one design, every segment resident
        {"name": "plate_3d", "kind": "plate3", "res": 64, "cx": 50, "cy": 10, "cz": 50, "tasks": 3, "steps": 100, "every": 50},
        # a small 3D walker on an odd grid: a design gradient early in a coarse-to-fine search
        {"name": "walker_3d_small", "kind": "walker3", "scale": 0.4, "steps": 100, "every": 50},
        # the 3D locomotion body (1,000,000 particles, 128^3): one checkpointed design gradient
        {"name": "walker_3d", "kind": "walker3", "scale": 1.0, "steps": 100, "every": 50},
        # the same body rolled out and its final state read back (no gradient)
        {"name": "rollout_3d", "kind": "rollout3", "scale": 1.0, "steps": 100, "every": 100},
        # a 3D plate in the non-uniform field of a permanent magnet
        {"name": "gradient_3d", "kind": "gradient3", "res": 48, "cx": 36, "cy": 8, "cz": 36, "tasks": 1, "steps": 50, "every": 25},
        # design maps, their reverse and the Adam steps of one design iteration (the 3D plate's particles)
        {"name": "design_3d", "kind": "design", "res": 64, "cx": 50, "cy": 10, "cz": 50, "tasks": 3, "steps": 1000, "radius": 1.5},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["substep", "beam", "rollout2", "walker2", "batch2", "clamp2", "plate3", "walker3", "walker3",
                       "rollout3", "gradient3", "design"])
    if kind == "substep":
        dim = rng.choice([2, 3])
        return {"kind": kind, "dim": dim, "res": rng.randint(24, 400) if dim == 2 else rng.randint(20, 64),
                "per_axis": rng.randint(2, 4) if dim == 2 else 2}
    if kind == "beam":
        return {"kind": kind, "res": rng.randint(32, 96), "per_axis": rng.randint(2, 4), "steps": rng.randint(50, 250)}
    if kind in ("rollout2", "walker2", "clamp2"):
        steps = rng.randint(100, 400)
        return {"kind": kind, "scale": round(rng.uniform(0.25, 1.0), 3), "steps": steps, "every": rng.choice([50, 100, steps])}
    if kind == "batch2":
        lo = log_int(500, 5000)
        return {"kind": kind, "instances": log_int(3, 64), "n_lo": lo, "n_hi": 8 * lo, "steps": rng.randint(40, 100),
                "every": rng.choice([25, 50])}
    if kind in ("plate3", "gradient3", "design"):
        res = rng.randint(28, 64 if kind != "gradient3" else 48)
        return {"kind": kind, "res": res, "cx": rng.randint(res // 3, (res * 25) // 32), "cy": rng.randint(4, 10),
                "cz": rng.randint(res // 3, (res * 25) // 32), "tasks": 1 if kind == "gradient3" else rng.randint(1, 3),
                **({"steps": rng.randint(200, 5000), "radius": round(rng.uniform(1.2, 2.5), 2)} if kind == "design" else
                   {"steps": rng.randint(20, 60), "every": rng.choice([10, 25, 60])})}
    steps = rng.randint(20, 100)
    return {"kind": kind, "scale": round(math.exp(rng.uniform(math.log(0.2), 0.0)), 3), "steps": steps,
            "every": rng.choice([20, 50, steps])}


# ---------------------------------------------------------------------------
# the workload (host arrays) behind a simulation case
# ---------------------------------------------------------------------------

def _grid_for(scale):
    # the grid that keeps the full-size body's share of the domain
    return max(28, int(round(128 * scale)))


def _batch_scales(c):
    # sizes spread evenly over [n_lo, n_hi], uneven from one instance to the next
    n = np.random.default_rng(c["instances"]).uniform(c["n_lo"], c["n_hi"], size=c["instances"])
    return [float(math.sqrt(k / 30000.0)) for k in n]


def _workload(c, seed):
    kind = c["kind"]
    if kind == "beam":
        return W.beam_2d(seed, per_axis=c["per_axis"], n_steps=c["steps"], res=c["res"])
    if kind in ("rollout2", "walker2", "clamp2"):
        s = c["scale"]
        w = W.walker_2d(seed, n_steps=c["steps"], res=_grid_for(s), scale=s, checkpoint_every=c["every"])
        if kind == "clamp2":
            x0, dx, dt = w.x0, 1.0 / w.cfg.res, w.cfg.dt
            top, left = float(x0[1].max()), float(x0[0].min())
            rng = np.random.default_rng([seed, 1])
            w.cfg.boundaries = [(B.MPM_BOUNDARY_ATTACHED, 0.0, (0.0, top - 1.37 * dx), (1.0, 1.0)),
                                (B.MPM_BOUNDARY_COULOMB, 0.4, (0.0, 0.0), (left + 3.71 * dx, 4.6 * dx))]
            t = np.arange(c["steps"]) * dt
            vel = rng.uniform(-0.05, 0.05, size=2)
            m = np.zeros((2, c["steps"], 2, 2), np.float32)
            m[0, :, 0] = (t[:, None] * vel[None]).astype(np.float32)
            m[0, :, 1] = vel
            w.bmotion = m
        return w
    if kind == "batch2":
        seeds = np.random.default_rng([seed, 5]).integers(1 << 30, size=c["instances"])
        return W.batch([W.walker_2d(int(s), n_steps=c["steps"], scale=k, checkpoint_every=c["every"])
                        for s, k in zip(seeds, _batch_scales(c))])
    if kind in ("plate3", "gradient3"):
        w = W.plate_3d(seed, n_steps=c["steps"], res=c["res"], n_tasks=c["tasks"], cells=(c["cx"], c["cy"], c["cz"]))
        w.cfg.checkpoint_every = c["every"]
        if kind == "gradient3":
            rng = np.random.default_rng([seed, 2])
            w.fgrad = (rng.uniform(-1, 1, size=(c["tasks"], 1, 3, 3)) *
                       np.cos(np.arange(c["steps"]) / 40.0)[None, :, None, None] * 0.05).astype(np.float32)
        return w
    s = c["scale"]
    return W.walker_3d(seed, n_steps=c["steps"], res=_grid_for(s), scale=s, checkpoint_every=c["every"])


def _gpu(a):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _substep_inputs(c, seed):
    """A body in motion: positions, velocities, affine matrices and strains."""
    d, res = c["dim"], c["res"]
    w = (W.beam_2d(seed, per_axis=c["per_axis"], n_steps=1, res=res) if d == 2 else
         W.plate_3d(seed, n_steps=1, res=res, n_tasks=1, cells=(res // 2, max(4, res // 8), res // 2)))
    rng = np.random.default_rng([seed, 3])
    n = w.x0.shape[1]
    state = np.concatenate([w.x0, 0.1 * rng.normal(size=(d, n)), rng.normal(size=(d * d, n)),
                            0.01 * rng.normal(size=(d * d, n))]).astype(np.float32)
    w.phi[:] = rng.uniform(0.2, 1.0, size=n)
    return w, state


DESIGN = {"Br_max": 0.1, "B_max": 0.02, "f_min": 1.0, "f_max": 20.0, "delta": 1e-6}


def _design_inputs(c, seed):
    """Design variables in the middle of an optimisation, upstream gradients, Adam moments."""
    rng = np.random.default_rng([seed, 4])
    w = W.plate_3d(seed, n_steps=1, res=c["res"], n_tasks=1, cells=(c["cx"], c["cy"], c["cz"]))
    n, t, d = w.x0.shape[1], c["tasks"], 3
    p = {"phi": rng.uniform(0.0, 1.0, n), "Br": rng.uniform(0.3, 1.0, n), "zeta": rng.uniform(-1, 1, (d, n)),
         "Ba": rng.uniform(0.2, 0.8, t), "f": rng.uniform(0.2, 0.8, t), "eta": rng.uniform(-1, 1, (t, d))}
    g = {"phi_bar": rng.normal(size=n), "mag": rng.normal(size=(d, n)), "field": rng.normal(size=(t, c["steps"], d))}
    f32 = {k: v.astype(np.float32) for k, v in p.items()}
    m = {k: (0.1 * rng.normal(size=v.shape)).astype(np.float32) for k, v in p.items()}
    s = {k: rng.uniform(0.5, 1.5, size=v.shape).astype(np.float32) for k, v in p.items()}
    return w.x0, f32, {k: v.astype(np.float32) for k, v in g.items()}, m, s


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------

BETA, LR, FIRST_K, DESIGN_DT = 8.0, 0.01, 10, 1.0e-4


def prepare(case, seed):
    kind = case["kind"]
    if kind == "substep":
        w, state = _substep_inputs(case, seed)
        c = B.mpm_config()
        counts = (ctypes.c_int * 1)(w.cfg.n_total)
        c.dim, c.grid_res, c.dt, c.n_steps = w.cfg.dim, w.cfg.res, w.cfg.dt, w.cfg.n_steps
        c.n_instances, c.n_particles, c.n_designs = 1, ctypes.cast(counts, B.P_int), 1
        c.E, c.nu, c.rho0, c.p_vol = w.cfg.E, w.cfg.nu, w.cfg.rho0, w.cfg.p_vol
        c.simp_eps, c.simp_q, c.damping_c = w.cfg.simp_eps, w.cfg.simp_q, w.cfg.damping
        for i in range(3):
            c.gravity[i] = w.cfg.gravity[i]
        c.bound, c.wall_mode, c.floor_mu, c.loss_kind = w.cfg.bound, w.cfg.wall_mode, w.cfg.floor_mu, w.cfg.loss_kind
        return {"kind": kind, "lib": B.load(), "cfg": c, "counts": counts, "state": _gpu(state), "phi": _gpu(w.phi),
                "mag": _gpu(w.mag), "field": _gpu(w.field[0])}
    if kind == "design":
        x0, p, g, m, s = _design_inputs(case, seed)
        maps = DesignMaps(_gpu(x0), case["tasks"], case["steps"], DESIGN_DT, case["radius"] / case["res"], **DESIGN)
        to = lambda t: {k: _gpu(v) for k, v in t.items()}  # noqa: E731
        return {"kind": kind, "maps": maps, "p": to(p), "g": to(g), "m": to(m), "v": to(s), "k": FIRST_K}
    w = _workload(case, seed)
    options = {}
    if kind == "batch2":  # what mpm_autotune picks for the batch of 64
        options = {B.MPM_OPT_SCATTER_2D: 1, B.MPM_OPT_ADJOINT_BLOCKS: 4}
    if kind == "plate3":
        options = {B.MPM_OPT_RESIDENT_SEGMENTS: -(-case["steps"] // case["every"])}
    sim = Simulator(w.cfg, options=options)
    if w.bmotion is not None:
        sim.set_boundaries(w.cfg.boundaries, _gpu(w.bmotion))
    if w.fgrad is not None:
        sim.set_field_gradient(_gpu(w.fgrad))
    if kind == "rollout2":  # host buffers, pinned as the entry point advises
        pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()  # noqa: E731
        return {"kind": kind, "sim": sim, "x0": pin(w.x0), "phi": pin(w.phi), "mag": pin(w.mag), "field": pin(w.field),
                "x": torch.empty(w.x0.shape).pin_memory(), "loss": torch.empty(1).pin_memory()}
    return {"kind": kind, "sim": sim, "x0": _gpu(w.x0), "phi": _gpu(w.phi), "mag": _gpu(w.mag), "field": _gpu(w.field),
            "target": _gpu(w.target), "one": torch.ones(w.cfg.n_instances, device="cuda")}


def run(state):
    s, kind = state, state["kind"]
    if kind == "substep":
        out = torch.empty_like(s["state"])
        st = s["lib"].mpm_substep_noalloc(ctypes.byref(s["cfg"]), 0, B.fptr(s["state"]), B.fptr(s["phi"]),
                                          B.fptr(s["mag"]), B.fptr(s["field"]), B.fptr(out),
                                          ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if st != B.MPM_OK:
            raise B.MpmError(st, (s["lib"].mpm_noalloc_last_error() or b"").decode())
        return {"state": out}
    if kind == "design":
        maps, p = s["maps"], s["p"]
        phi_bar, mag, field = maps.forward(p, BETA)
        grads = maps.backward(s["g"]["phi_bar"], s["g"]["mag"], s["g"]["field"])
        for name, x in p.items():
            lo, hi = PARAM_BOX[name]
            adam_step(x, grads[name], s["m"][name], s["v"][name], s["k"], LR, lo, hi)
        s["k"] += 1
        return {"phi_bar": phi_bar, "mag": mag, "field": field, "grads": grads, "params": p, "m": s["m"], "v": s["v"]}
    sim = s["sim"]
    if kind == "rollout2":
        sim.forward_host(s["x0"], s["phi"], s["mag"], s["field"], x_out=s["x"], loss_out=s["loss"])
        return {"loss": s["loss"], "x": s["x"]}
    if kind == "rollout3":
        loss, x = sim.forward(s["x0"], s["phi"], s["mag"], s["field"], want_x=True)
        u, v, C, E = sim.read_state_strain()
        return {"loss": loss, "x": x, "u": u, "v": v, "C": C, "E": E}
    if kind == "beam":
        phi, mag, field = (s[k].detach().requires_grad_(True) for k in ("phi", "mag", "field"))
        loss = MpmSim.apply(sim, s["x0"], phi, mag, field, s["target"], None)
        loss.sum().backward()
        return {"loss": loss.detach(), "g_phi": phi.grad, "g_mag": mag.grad, "g_field": field.grad}
    loss, _ = sim.forward(s["x0"], s["phi"], s["mag"], s["field"], target=s["target"])
    g_phi, g_mag, g_field = sim.backward(s["one"])
    out = {"loss": loss, "g_phi": g_phi, "g_mag": g_mag, "g_field": g_field}
    if kind == "gradient3":
        out["g_fgrad"] = sim.field_gradient_grad()
    return out


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

def _body_particles(c):
    """Particles of all instances of a case."""
    kind = c["kind"]
    if kind == "batch2":
        return sum(_body_particles({"kind": "walker2", "scale": s}) for s in _batch_scales(c))
    if kind in ("rollout2", "walker2", "clamp2"):
        s = c["scale"]
        tw, th = max(8, int(round(100 * s))), max(4, int(round(45 * s)))
        lw, lh = max(2, int(round(15 * s))), max(2, int(round(50 * s)))
        return 4 * (tw * th + 4 * lw * lh)
    if kind in ("walker3", "rollout3"):
        s = c["scale"]
        tw, th, td = max(6, int(round(100 * s))), max(3, int(round(25 * s))), max(3, int(round(40 * s)))
        lw, lh, ld = max(2, int(round(10 * s))), max(2, int(round(25 * s))), max(2, int(round(25 * s)))
        return 8 * (tw * th * td + 4 * lw * lh * ld)
    if kind == "beam" or (kind == "substep" and c["dim"] == 2):
        return int(round(0.5 * c["res"])) * int(round(0.125 * c["res"])) * c["per_axis"] ** 2
    if kind == "substep":
        return 8 * (c["res"] // 2) ** 2 * max(4, c["res"] // 8)
    return 8 * c["cx"] * c["cy"] * c["cz"] * (1 if kind == "design" else c["tasks"])


def work(case):
    """Per particle and substep, as a horizon's states do not fit on the chip:
    the forward reads and writes the state (x, v, C, F) once and reads the
    design; the adjoint reads the stored state and the adjoint of n + 1,
    writes that of n, and reads and updates the design and its gradients; each
    passes over the touched nodes (one per 4 / 8 particles) once.  Operations
    are those of the stencil sums (9 / 27 nodes) and the stress."""
    kind = case["kind"]
    n = _body_particles(case)
    if kind == "design":
        d, r = 3, case["radius"]
        # two filter passes over the neighbours inside the radius (8 particles per cell)
        near = 8 * 4.0 / 3.0 * math.pi * r ** 3
        per = 4 * (d + 2 * (1 + d) + 3 * 4 * (1 + 1 + d) + (1 + d)) + 4 * 2
        return {"bytes": float(n * per + 8 * case["tasks"] * case["steps"] * d), "flops": float(n * (2 * near * 12 + 150))}
    d = 2 if kind in ("rollout2", "walker2", "clamp2", "beam", "batch2") else 3
    if kind == "substep":
        d = case["dim"]
    fwd, adj = ((118, 200) if d == 2 else (215, 350))
    f_ops, a_ops = ((550, 1300) if d == 2 else (1600, 3700))
    steps = 1 if kind == "substep" else case["steps"]
    grad = kind not in ("substep", "rollout2", "rollout3")
    return {"bytes": float(n * steps * (fwd + (adj if grad else 0))), "flops": float(n * steps * (f_ops + (a_ops if grad else 0)))}


# ---------------------------------------------------------------------------
# exact: the method in plain torch, 64 bits, reverse mode by autograd
# ---------------------------------------------------------------------------

class _Exact:
    """MLS-MPM of hard-magnetic material on [N, d] float64 tensors."""

    def __init__(self, w):
        self.w, self.cfg = w, w.cfg
        c = w.cfg
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        d = self.d = c.dim
        self.nodes = c.res ** d
        counts = torch.tensor(c.counts, device=self.dev)
        self.inst = torch.repeat_interleave(torch.arange(len(c.counts), device=self.dev), counts)
        first = np.concatenate([[0], np.cumsum(c.design_counts())])
        self.design = torch.cat([torch.arange(n, device=self.dev) + int(first[z]) for n, z in zip(c.counts, c.designs)])
        self.G = c.E / (2 * (1 + c.nu))
        self.K = c.E / (3 * (1 - 2 * c.nu))
        o = torch.arange(3, device=self.dev)
        self.off = torch.cartesian_prod(*([o] * d))  # [3^d, d], last axis fastest
        g = torch.arange(c.res, device=self.dev)
        self.coord = torch.cartesian_prod(*([g] * d))  # [nodes, d]
        self.stride = torch.tensor([c.res ** (d - 1 - a) for a in range(d)], device=self.dev)

    def f64(self, a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(self.dev)

    def stencil(self, x):
        c = self.cfg
        fx = x * c.res
        base = torch.floor(fx.detach() - 0.5)
        r = fx - base
        w1 = torch.stack([0.5 * (1.5 - r) ** 2, 0.75 - (r - 1) ** 2, 0.5 * (r - 0.5) ** 2], dim=-1)  # [N, d, 3]
        w = w1[:, 0, :].index_select(1, self.off[:, 0])
        for a in range(1, self.d):
            w = w * w1[:, a, :].index_select(1, self.off[:, a])
        dpos = (self.off[None].to(x.dtype) - r[:, None, :]) / c.res
        node = ((base.long()[:, None, :] + self.off[None]) * self.stride).sum(-1) + self.inst[:, None] * self.nodes
        return w, dpos, node

    def stress(self, F, phi, mag, Bp):
        c, d = self.cfg, self.d
        J = torch.linalg.det(F)
        H = torch.linalg.inv(F).transpose(1, 2)
        I1 = (F * F).sum((1, 2)) + (1.0 if d == 2 else 0.0)
        col = lambda t: t[:, None, None]  # noqa: E731
        Pe = col(self.G * J ** (-2.0 / 3.0)) * (F - col(I1 / 3) * H) + col(self.K * J * (J - 1)) * H
        s = phi ** c.simp_q
        return col(c.simp_eps + (1 - c.simp_eps) * s) * Pe - col(s / MU0) * Bp[:, :, None] * mag[:, None, :]

    def grid(self, m, mv, n):
        c, d = self.cfg, self.d
        live = m > 0
        ms = torch.where(live, m, torch.ones_like(m))
        g = torch.tensor(list(c.gravity)[:d], dtype=m.dtype, device=self.dev)
        v = torch.where(live[:, None], (1 - c.dt * c.damping) * mv / ms[:, None] + c.dt * g, torch.zeros_like(mv))
        coord = self.coord.repeat(len(c.counts), 1)

        def coulomb(r, axis, sgn, mu):  # r: velocity relative to the boundary
            keep = torch.ones(d, dtype=r.dtype, device=self.dev)
            keep[axis] = 0
            t = r * keep
            t2 = (t * t).sum(-1)
            u = torch.sqrt(torch.where(t2 > 0, t2, torch.ones_like(t2)))
            sp = u + mu * sgn * r[:, axis]
            f = torch.where((t2 > 0) & (sp > 0), sp / u, torch.zeros_like(u))
            return t * f[:, None]

        for a in range(d):
            for side in (0, 1):
                band = coord[:, a] < c.bound if side == 0 else coord[:, a] >= c.res - c.bound
                hit = (band & ((v[:, a] if side == 0 else -v[:, a]) < 0))[:, None]
                if c.wall_mode == 1 and a == 1 and side == 0:
                    v = torch.where(hit, coulomb(v, 1, 1.0, c.floor_mu), v)
                else:
                    v = torch.where(hit, torch.zeros_like(v), v)
        for b, (kind, mu, lo, hi) in enumerate(c.boundaries or []):
            mo = np.zeros((2, d)) if self.w.bmotion is None else self.w.bmotion[b, n].astype(np.float64)
            vb = torch.tensor(mo[1], dtype=v.dtype, device=self.dev)
            x = coord.to(v.dtype) / c.res
            l = torch.tensor(np.float32(lo)[:d].astype(np.float64) + mo[0], device=self.dev)
            h = torch.tensor(np.float32(hi)[:d].astype(np.float64) + mo[0], device=self.dev)
            inside = ((x >= l) & (x <= h)).all(-1)
            dist = torch.stack([x - l, h - x], dim=-1).reshape(x.shape[0], 2 * d)  # low face of axis 0, high, ...
            face = dist.argmin(-1)
            rel = v - vb
            sgn = (2 * (face % 2) - 1).to(v.dtype)
            into = sgn * rel.gather(1, (face // 2)[:, None])[:, 0] < 0
            if kind == B.MPM_BOUNDARY_COULOMB:
                for a in range(d):
                    hit = inside & into & (face // 2 == a)
                    v = torch.where(hit[:, None], vb + coulomb(rel, a, sgn, float(np.float32(mu))), v)
            else:
                hit = inside if kind == B.MPM_BOUNDARY_ATTACHED else inside & into
                v = torch.where(hit[:, None], vb.expand_as(v), v)
        return v

    def substep(self, n, x, v, C, F, phi, mag, B_n, G_n):
        c, d = self.cfg, self.d
        dt, kappa = c.dt, 4.0 * c.res * c.res
        mp = phi * c.rho0 * c.p_vol
        Bp = B_n[self.inst]
        mom = mp[:, None] * v
        if G_n is not None:
            Gp = G_n[self.inst]
            Bp = Bp + (Gp @ (x - 0.5)[:, :, None])[:, :, 0]
            FB = F @ mag[:, :, None]
            f = (phi ** c.simp_q * c.p_vol / MU0)[:, None] * (Gp.transpose(1, 2) @ FB)[:, :, 0]
            mom = mom + dt * f
        P = self.stress(F, phi, mag, Bp)
        A = mp[:, None, None] * C - dt * kappa * c.p_vol * P @ F.transpose(1, 2)
        w, dpos, node = self.stencil(x)
        val = torch.cat([mp[:, None, None].expand(-1, w.shape[1], 1), mom[:, None, :] + dpos @ A.transpose(1, 2)], dim=-1)
        grid = torch.zeros(self.nodes * len(c.counts), 1 + d, dtype=x.dtype, device=self.dev)
        grid = grid.index_add(0, node.reshape(-1), (w[:, :, None] * val).reshape(-1, 1 + d))
        V = self.grid(grid[:, 0], grid[:, 1:], n)
        wv = w[:, :, None] * V.index_select(0, node.reshape(-1)).reshape(*node.shape, d)
        v = wv.sum(1)
        C = kappa * wv.transpose(1, 2) @ dpos
        x = x + dt * v
        F = F + dt * C @ F
        return x, v, C, F

    def simulate(self, grad):
        w, c, d = self.w, self.cfg, self.d
        x0 = self.f64(w.x0.T)
        phi, mag, field = (self.f64(a).requires_grad_(grad) for a in (w.phi, w.mag, w.field))
        fg = None if w.fgrad is None else self.f64(w.fgrad).requires_grad_(grad)
        phi_p, mag_p = phi[self.design], mag.T[self.design]
        x, v = x0, torch.zeros_like(x0)
        C = torch.zeros(x0.shape[0], d, d, dtype=torch.float64, device=self.dev)
        F = torch.eye(d, dtype=torch.float64, device=self.dev).expand_as(C).contiguous()
        mp = phi_p * c.rho0 * c.p_vol
        ni = len(c.counts)
        total = lambda t: torch.zeros(ni, dtype=t.dtype, device=self.dev).index_add(0, self.inst, t)  # noqa: E731
        M, loss = total(mp), torch.zeros(ni, dtype=torch.float64, device=self.dev)
        for n in range(c.n_steps):
            args = (n, x, v, C, F, phi_p, mag_p, field[:, n], None if fg is None else fg[:, n])
            x, v, C, F = (checkpoint(self.substep, *args, use_reentrant=False, preserve_rng_state=False) if grad
                          else self.substep(*args))
            if c.loss_kind == 1:
                loss = loss - c.dt * total(mp * v[:, 0]) / M
        if c.loss_kind == 0:
            cnt = torch.tensor(c.counts, dtype=torch.float64, device=self.dev)
            loss = total(((x - self.f64(w.target.T)) ** 2).sum(-1)) / cnt
        if not grad:
            eye = torch.eye(d, dtype=torch.float64, device=self.dev)
            flat = lambda t: t.permute(1, 2, 0)  # noqa: E731
            return {"loss": loss, "x": x.T, "u": (x - x0).T, "v": v.T, "C": flat(C), "E": flat(F - eye)}
        loss.sum().backward()
        out = {"loss": loss.detach(), "g_phi": phi.grad, "g_mag": mag.grad, "g_field": field.grad}
        if fg is not None:
            out["g_fgrad"] = fg.grad
        return out


def _exact_design(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x0, p, g, m, s = _design_inputs(case, seed)
    f64 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to(dev)  # noqa: E731
    X = f64(x0).T.contiguous()
    R = case["radius"] / case["res"]
    order = torch.argsort(X[:, 0])
    xs = X[order]

    def filt(vals):  # sum_q (1 - |x_q - x_p| / R) vals_q over |x_q - x_p| < R, [N, k]
        vs, out = vals[order], torch.empty_like(vals)
        for i in range(0, xs.shape[0], 2048):
            a = xs[i:i + 2048]
            lo = int(torch.searchsorted(xs[:, 0].contiguous(), a[0, 0] - R))
            hi = int(torch.searchsorted(xs[:, 0].contiguous(), a[-1, 0] + R))
            d2 = torch.zeros(a.shape[0], hi - lo, dtype=torch.float64, device=dev)
            for k in range(3):
                d2 += (a[:, k, None] - xs[None, lo:hi, k]) ** 2
            out[order[i:i + 2048]] = torch.clamp(1 - torch.sqrt(d2) / R, min=0) @ vs[lo:hi]
        return out

    P = {k: f64(v).requires_grad_(True) for k, v in p.items()}
    norm = filt(torch.ones_like(X[:, :1]))[:, 0]
    phi_t = (filt(P["phi"].detach()[:, None])[:, 0] / norm).requires_grad_(True)
    th = math.tanh(BETA * 0.5)
    phi_bar = (th + torch.tanh(BETA * (phi_t - 0.5))) / (2 * th)
    unit = lambda z, dim: z / torch.sqrt((z * z).sum(dim, keepdim=True) + DESIGN["delta"])  # noqa: E731
    mag = DESIGN["Br_max"] * P["Br"] * unit(P["zeta"], 0)
    fbar = (DESIGN["f_max"] - DESIGN["f_min"]) * P["f"] + DESIGN["f_min"]
    t = torch.arange(case["steps"], dtype=torch.float64, device=dev) * DESIGN_DT
    wave = DESIGN["B_max"] * P["Ba"][:, None] * torch.sin(2 * math.pi * fbar[:, None] * t)
    field = wave[:, :, None] * unit(P["eta"], 1)[:, None, :]
    ((phi_bar * f64(g["phi_bar"])).sum() + (mag * f64(g["mag"])).sum() + (field * f64(g["field"])).sum()).backward()
    grads = {k: v.grad for k, v in P.items()}
    grads["phi"] = filt((phi_t.grad / norm)[:, None])[:, 0]
    new, m1, v1 = {}, {}, {}
    for k, v in P.items():
        m1[k] = 0.9 * f64(m[k]) + 0.1 * grads[k]
        v1[k] = 0.999 * f64(s[k]) + 0.001 * grads[k] ** 2
        step = LR * (m1[k] / (1 - 0.9 ** FIRST_K)) / (torch.sqrt(v1[k] / (1 - 0.999 ** FIRST_K)) + 1e-8)
        new[k] = torch.clamp(v.detach() - step, *PARAM_BOX[k])
    return {"phi_bar": phi_bar.detach(), "mag": mag.detach(), "field": field.detach(), "grads": grads, "params": new,
            "m": m1, "v": v1}


def exact(case, seed):
    kind = case["kind"]
    if kind == "design":
        return _exact_design(case, seed)
    if kind == "substep":
        w, state = _substep_inputs(case, seed)
        e = _Exact(w)
        d, s = e.d, e.f64(state)
        n = s.shape[1]
        mat = lambda t: t.reshape(d, d, n).permute(2, 0, 1)  # noqa: E731
        eye = torch.eye(d, dtype=torch.float64, device=e.dev)
        x, v, C, F = e.substep(0, s[:d].T, s[d:2 * d].T, mat(s[2 * d:2 * d + d * d]), mat(s[2 * d + d * d:]) + eye,
                               e.f64(w.phi), e.f64(w.mag.T), e.f64(w.field[:, 0]), None)
        flat = lambda t: t.permute(1, 2, 0).reshape(d * d, n)  # noqa: E731
        return {"state": torch.cat([x.T, v.T, flat(C), flat(F - eye)])}
    e = _Exact(_workload(case, seed))
    if kind in ("rollout2", "rollout3"):
        out = e.simulate(False)
        return out if kind == "rollout3" else {"loss": out["loss"], "x": out["x"]}
    return e.simulate(True)
