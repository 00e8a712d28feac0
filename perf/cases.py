"""The work that users have this framework do, as cases that can be timed.

Five kinds of call, each through the public entry points:

  job         a simulation from its workload to its results: the context is
              built, the particles added, `steps` steps run, the fields and the
              particle state of every instance read, the context closed (what a
              script, a parameter study or a data-generation loop does);
  frames      a context that is kept: it is set back to a saved state, advances
              and hands out its particles every few steps (a recorded
              trajectory, a restart, a control loop);
  gradient    the differentiable trajectory (paper_2511_01629_gb300.autograd): a
              forward pass with checkpoints and its backward, with torch
              parameters in torch's default type;
  fields      the macroscopic fields of a running simulation written to device
              tensors (a movie frame, a training sample);
  projection  the rigid-body projection of a velocity field that the caller
              holds, by the allocation-free entry point of the C ABI.

`exact` is the method of the paper (Eqs. 9-22, Algorithm 1) in plain torch, in
64 bits: a dense pull-scheme lattice step, the solid nodes recomputed with
their force and penalty, and the particle update.  Gradients come from
torch's reverse mode with the solid domains held fixed.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2511_01629_gb300 import autograd, lbm
from paper_2511_01629_gb300 import workloads as W

_STORAGE = {"fp32": lbm.LBM_FP32, "fp16": lbm.LBM_FP16}
_EXACT_NODE_STEPS = 1.2e10  # beyond this the 64-bit run takes over about 20 s


# ------------------------------------------------------------------ cases ---
def listed():
    return [
        # the paper's channel test: a neutrally buoyant disk in Poiseuille flow, periodic in x,
        # tau = 0.8; the smallest grid, run to its full horizon of 2000 steps
        {"name": "channel_100x200", "kind": "job", "scene": "channel", "nx": 100, "ny": 200, "steps": 2000,
         "storage": "fp32", "K": 1},
        # one settling disk (Sec. 3.2), its trajectory recorded every 10 steps from a restart
        {"name": "frames_disk_400x1600", "kind": "frames", "scene": "disk", "nx": 400, "ny": 1600, "frames": 80,
         "every": 10, "storage": "fp32", "K": 1},
        # the many-particle case (Sec. 3.5), the framework's headline workload, in both storage types
        {"name": "disks500_fp32", "kind": "job", "scene": "disks", "nx": 1024, "ny": 4096, "np": 500, "steps": 600,
         "storage": "fp32", "K": 1},
        {"name": "disks500_fp16", "kind": "job", "scene": "disks", "nx": 1024, "ny": 4096, "np": 500, "steps": 600,
         "storage": "fp16", "K": 1},
        # 64 independent boxes of ragged sizes in one context: the largest call
        {"name": "ensemble_64", "kind": "job", "scene": "ensemble", "count": 64, "nx_lo": 200, "nx_hi": 800,
         "np_hi": 50, "steps": 120, "storage": "fp32", "K": 1},
        # the 3D workload: eight spheres settling in a closed box
        {"name": "spheres_256x256x512", "kind": "job", "scene": "spheres", "nx": 256, "ny": 256, "nz": 512, "np": 8,
         "radius": 10.0, "steps": 60, "storage": "fp32", "K": 1},
        # 3D in 16-bit storage with odd sizes on every axis
        {"name": "spheres_fp16_ragged", "kind": "job", "scene": "spheres", "nx": 151, "ny": 133, "nz": 203, "np": 5,
         "radius": 8.0, "steps": 160, "storage": "fp16", "K": 1},
        # lateral migration in plane Couette flow (Sec. 3.1): moving walls, periodic in x, a large disk
        {"name": "couette_5000x200", "kind": "job", "scene": "couette", "H": 200, "diameter": 50.0, "length_d": 100.0,
         "steps": 600, "storage": "fp32", "K": 1},
        # the adjoint workload: one settling disk, then sixteen seeds in one context
        {"name": "gradient_disk", "kind": "gradient", "nx": 400, "ny": 1600, "nz": 1, "batch": 1, "np": 1,
         "radius": 12.0, "steps": 240, "storage": "fp32"},
        {"name": "gradient_batch16", "kind": "gradient", "nx": 400, "ny": 1600, "nz": 1, "batch": 16, "np": 1,
         "radius": 12.0, "steps": 48, "storage": "fp32"},
        # one frame of the many-particle case
        {"name": "fields_disks500", "kind": "fields", "scene": "disks", "nx": 1024, "ny": 4096, "np": 500, "steps": 40,
         "storage": "fp32", "K": 1},
        # the shortest call: 500 disks projected out of a given field
        {"name": "projection_disks500", "kind": "projection", "scene": "disks", "nx": 1024, "ny": 4096, "np": 500},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_scene(rng, projection=False):
    s = rng.choice(["disk", "disks", "disks", "spheres", "spheres"] if projection else
                   ["channel", "disk", "disks", "disks", "spheres", "spheres", "couette", "ellipse"])
    if s == "channel":
        return {"scene": s, "nx": _log(rng, 64, 800), "ny": _log(rng, 64, 800)}
    if s == "disk":
        nx = _log(rng, 80, 700)
        return {"scene": s, "nx": nx, "ny": rng.randint(2 * nx, 4 * nx)}
    if s == "disks":
        nx, ny = _log(rng, 128, 1024), _log(rng, 256, 4096)
        return {"scene": s, "nx": nx, "ny": ny, "np": _log(rng, 2, max(3, nx * ny // 8400))}
    if s == "spheres":
        n = [_log(rng, 48, 200) for _ in range(3)]
        return {"scene": s, "nx": n[0], "ny": n[1], "nz": n[2], "np": rng.randint(1, 6),
                "radius": round(rng.uniform(4.0, 8.0), 3)}
    if s == "couette":
        H = _log(rng, 60, 240)
        return {"scene": s, "H": H, "diameter": round(0.25 * H, 3), "length_d": float(rng.randint(20, 100))}
    return {"scene": "ellipse", "L": _log(rng, 60, 240)}


def draw(rng):
    kind = rng.choice(["job", "job", "job", "ensemble", "frames", "gradient", "fields", "projection"])
    if kind == "projection":
        return {"kind": kind, **_draw_scene(rng, projection=True)}
    if kind == "gradient":
        three = rng.random() < 0.3
        c = {"kind": kind, "batch": _log(rng, 1, 4 if three else 16), "np": rng.randint(1, 3),
             "steps": rng.randint(16, 96), "storage": rng.choice(["fp32", "fp32", "fp16"])}
        if three:
            c.update(nx=_log(rng, 40, 96), ny=_log(rng, 40, 96), nz=_log(rng, 64, 128), radius=round(rng.uniform(4, 7), 3))
            c["steps"] = min(c["steps"], 32)
        else:
            c["nx"] = _log(rng, 100, 400)
            c.update(ny=rng.randint(3 * c["nx"], 4 * c["nx"]), nz=1, radius=round(rng.uniform(5, 12), 3))
        return c
    storage = rng.choice(["fp32", "fp16"])
    if kind == "ensemble":
        lo = _log(rng, 100, 500)
        c = {"kind": "job", "scene": "ensemble", "count": _log(rng, 2, 64), "nx_lo": lo, "nx_hi": rng.randint(lo + 20, lo + 300),
             "np_hi": rng.randint(2, 20), "storage": storage, "K": 1}
        nodes = c["count"] * (lo + c["nx_hi"]) ** 2
    else:
        c = {"kind": kind, **_draw_scene(rng), "storage": storage, "K": rng.choice([1, 1, 1, 2])}
        nodes = math.prod(_sizes(c))
    steps = max(16, min(900, int(1.6e9 / (nodes * (2.2 if c["scene"] == "spheres" else 1.0)))))
    if kind == "frames":
        c["every"] = rng.choice([1, 4, 10, 20])
        c["frames"] = max(2, steps // c["every"])
    elif kind == "fields":
        c["steps"] = min(steps, 40)
    else:
        c["steps"] = steps
    return c


def _sizes(c):
    s = c["scene"]
    if s == "couette":
        return (int(round(c["length_d"] * c["diameter"])), c["H"], 1)
    if s == "ellipse":
        return (c["L"], 10 * c["L"], 1)
    return (c["nx"], c["ny"], c.get("nz", 1))


# ----------------------------------------------------------------- inputs ---
def _scene(c, seed):
    """The workloads (one per instance) of a case."""
    s, rng = c["scene"], np.random.default_rng([seed, 17])
    if s == "channel":
        ws = [W.poiseuille_disk(seed, c["nx"], c["ny"])]
    elif s == "disk":
        r = 12.0 if c["nx"] >= 200 else 6.0
        ws = [W.single_disk(seed, c["nx"], c["ny"], radius=r)]
    elif s == "disks":
        ws = [W.many_disks(seed, c["nx"], c["ny"], c["np"])]
    elif s == "ensemble":
        # the sizes are the case's, the particles the seed's (workloads.ensemble draws both from one seed)
        sizes = np.random.default_rng([c["count"], c["nx_lo"], c["nx_hi"]])
        ws = []
        for i in range(c["count"]):
            nx, n = int(sizes.integers(c["nx_lo"], c["nx_hi"] + 1)), int(sizes.integers(1, c["np_hi"] + 1))
            ws.append(W.many_disks(1000 * seed + i, nx, 4 * nx, n))
    elif s == "spheres":
        ws = [W.spheres3d(seed, c["nx"], c["ny"], c["nz"], c["np"], c["radius"])]
    elif s == "couette":
        w = W.couette_migration(c["H"], c["diameter"], c["length_d"])
        w.pos[0][0] += rng.uniform(-2.0, 2.0) * c["diameter"]
        w.pos[0][1] += rng.uniform(0.0, 1.0) * c["diameter"]
        ws = [w]
    else:
        w = W.ellipse_settling(c["L"], theta0=rng.uniform(0.1, 1.4))
        w.pos[0][0] += rng.uniform(-0.1, 0.1) * c["L"]
        ws = [w]
    for w in ws:
        w.K = c.get("K", 1)
    return ws


def _gradient_inputs(c, seed):
    """(alpha, ratio, X0, U0) and the incoming gradients (gX, gU), float32 on the host."""
    rng = np.random.default_rng([seed, 29])
    D = 3 if c["nz"] > 1 else 2
    B, P, r = c["batch"], c["np"], c["radius"]
    n = (c["nx"], c["ny"], c["nz"])
    X0 = np.zeros((B, P, D))
    for d in range(D):
        X0[:, :, d] = n[d] / 2 + rng.uniform(-0.05, 0.05, (B, P)) * n[d]
    gap = max(0.12 * n[D - 1], 2 * r + 5.0)  # stacked along gravity, clear of each other
    X0[:, :, D - 1] = 0.5 * n[D - 1] + (np.arange(P) - 0.5 * (P - 1)) * gap + rng.uniform(-0.5, 0.5, (B, P))
    f = lambda a: np.asarray(a, np.float32)
    return (f(rng.uniform(0.85, 1.0, B)), f(rng.uniform(1.1, 2.0, (B, P))), f(X0), f(rng.uniform(-1e-4, 1e-4, (B, P, D))),
            f(rng.normal(size=(B, P, D))), f(rng.normal(size=(B, P, D)) * 10.0))


def _gravity(D):
    return (0.0, -2e-6, 0.0) if D == 2 else (0.0, 0.0, -2e-6)


def _velocity(n, D, seed):
    """A smooth velocity field [D, nz, ny, nx] (float32) of the size that settling flows have."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    ax = [torch.linspace(0.0, 2.0 * math.pi, n[d], device="cuda") for d in (2, 1, 0)]
    zz, yy, xx = ax[0].view(-1, 1, 1), ax[1].view(1, -1, 1), ax[2].view(1, 1, -1)
    u = torch.empty((D, n[2], n[1], n[0]), dtype=torch.float32, device="cuda")
    for d in range(D):
        k = torch.rand(7, generator=g, device="cuda")
        u[d] = 0.02 * torch.sin((1 + 5 * k[0]) * xx + 6 * k[1]) * torch.cos((1 + 5 * k[2]) * yy + 6 * k[3]) * \
            torch.cos((1 + 5 * k[4]) * zz + 6 * k[5])
        u[d] += 1e-3 * (torch.rand(u[d].shape, generator=g, device="cuda") - 0.5)
    return u


class _Fields:
    """Device tensors for u, p and owner of every instance, kept by the caller."""

    def __init__(self, ws):
        self.D = ws[0].D
        self.nodes = [w.nodes for w in ws]
        N = sum(self.nodes)
        self.u = torch.empty(self.D * N, dtype=torch.float32, device="cuda")
        self.p = torch.empty(N, dtype=torch.float32, device="cuda")
        self.owner = torch.empty(N, dtype=torch.int32, device="cuda")

    def read(self, sim):
        o = 0
        for i, n in enumerate(self.nodes):
            sim.fields_device(i, self.u[self.D * o:self.D * (o + n)], self.p[o:o + n], self.owner[o:o + n])
            o += n
        return {"u": self.u, "p": self.p, "owner": self.owner}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        D = 3 if case["nz"] > 1 else 2
        al, ra, X0, U0, gX, gU = (torch.from_numpy(a).cuda() for a in _gradient_inputs(case, seed))
        walls = (lbm.LBM_WALL, lbm.LBM_WALL, lbm.LBM_WALL if D == 3 else lbm.LBM_PERIODIC)
        n = (case["nx"], case["ny"], case["nz"])[:D]
        make = autograd.sedimentation_factory(n, case["radius"], tau=1.0, g_grav=_gravity(D),
                                              storage=_STORAGE[case["storage"]], walls=walls)
        params = [t.requires_grad_(True) for t in (al, ra, X0, U0)]
        return {"kind": kind, "params": params, "seeds": (gX, gU), "factory": make, "steps": case["steps"]}
    ws = _scene(case, seed)
    if kind == "projection":
        w = ws[0]
        f64 = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")
        np_, D = w.num_particles, w.D
        return {"kind": kind, "D": D, "np": np_, "n": (ctypes.c_int * 3)(*w.n), "per": (ctypes.c_int * 3)(*w.periodic),
                "u": _velocity(w.n, D, seed), "pos": f64(w.pos).reshape(np_, D), "radius": f64(w.radius), "rmax": float(max(w.radius)),
                "vel": torch.empty((np_, D), dtype=torch.float64, device="cuda"),
                "omega": torch.empty((np_, 1 if D == 2 else 3), dtype=torch.float64, device="cuda"),
                "count": torch.empty(np_, dtype=torch.int32, device="cuda"), "call": _projection_entry()}
    st = {"kind": kind, "ws": ws, "storage": _STORAGE[case["storage"]]}
    if kind == "job":
        st.update(steps=case["steps"], fields=_Fields(ws))
        return st
    sim = lbm.from_workloads(ws, st["storage"])
    if kind == "fields":
        sim.step(case["steps"])
        sim.sync()
        st.update(sim=sim, fields=_Fields(ws))
        return st
    pin = lambda dt, *s: torch.empty(s, dtype=dt, pin_memory=True).numpy()
    F, n = case["frames"], ws[0].num_particles
    st.update(sim=sim, blob=sim.save_state(), every=case["every"],
              out={**{k: pin(torch.float64, F, n, 3) for k in ("X", "U", "W", "theta", "A")}, "count": pin(torch.int32, F, n)})
    return st


def _projection_entry():
    fn = lbm.lib().lbm_rigid_projection_noalloc
    v, ip = ctypes.c_void_p, ctypes.POINTER(ctypes.c_int)
    fn.restype = ctypes.c_int
    fn.argtypes = [ctypes.c_int, ip, ip, v, ctypes.c_int, v, v, ctypes.c_double, v, v, v, v]
    return fn


def run(state):
    kind = state["kind"]
    if kind == "job":
        sim = lbm.from_workloads(state["ws"], state["storage"])
        sim.step(state["steps"])
        out = state["fields"].read(sim)
        parts = [sim.particles(i) for i in range(len(state["ws"]))]
        for k in ("X", "U", "W", "theta", "A", "count"):
            out[k] = np.concatenate([q[k] for q in parts])
        sim.close()
        return out
    if kind == "frames":
        sim, out = state["sim"], state["out"]
        sim.load_state(state["blob"])
        for f in range(len(out["count"])):
            sim.step(state["every"])
            sim.particles_async({k: out[k][f] for k in out})
        sim.sync()
        return out
    if kind == "fields":
        return state["fields"].read(state["sim"])
    if kind == "gradient":
        X, U = autograd.trajectory(*state["params"], state["factory"], state["steps"])
        grads = torch.autograd.grad((X, U), state["params"], state["seeds"])
        return {"X": X, "U": U, "alpha": grads[0], "ratio": grads[1], "X0": grads[2], "U0": grads[3]}
    s, p = state, lambda t: ctypes.c_void_p(t.data_ptr())
    rc = s["call"](s["D"], s["n"], s["per"], p(s["u"]), s["np"], p(s["pos"]), p(s["radius"]), s["rmax"], p(s["vel"]),
                   p(s["omega"]), p(s["count"]), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if rc != 0:
        raise RuntimeError(f"lbm_rigid_projection_noalloc: {rc}")
    return {"vel": s["vel"], "omega": s["omega"], "count": s["count"]}


def work(case):
    """Bytes and operations of one pass.  A step reads and writes every moving
    population once; the adjoint of a step reads the populations entering it
    and the adjoint field and writes the adjoint field (FP32)."""
    kind = case["kind"]
    if kind == "gradient":
        three = case["nz"] > 1
        q, s = (18, 330) if three else (8, 130)
        e = 2 if case["storage"] == "fp16" else 4
        node_steps = case["batch"] * case["nx"] * case["ny"] * case["nz"] * case["steps"]
        return {"bytes": node_steps * q * (3 * e + 8), "flops": node_steps * 4 * s}
    if kind == "projection":
        ws = _scene(case, 0)
        D = ws[0].D
        solid = sum(math.pi * r * r if D == 2 else 4.0 / 3.0 * math.pi * r ** 3 for r in ws[0].radius)
        return {"bytes": solid * 4 * D + 8.0 * ws[0].num_particles * (2 * D + 4), "flops": solid * 20 * D}
    e = 2 if case["storage"] == "fp16" else 4
    if case["scene"] == "ensemble":
        nodes, q, s, d = sum(w.nodes for w in _scene(case, 0)), 8, 130, 2
    else:
        nodes = math.prod(_sizes(case))
        q, s, d = (18, 330, 3) if case["scene"] == "spheres" else (8, 130, 2)
    out = nodes * 4 * (d + 2)
    if kind == "fields":
        return {"bytes": nodes * q * e + out, "flops": nodes * 4 * q}
    steps = case["frames"] * case["every"] if kind == "frames" else case["steps"]
    return {"bytes": steps * nodes * 2 * q * e + (out if kind == "job" else nodes * q * e), "flops": steps * nodes * s}


# ------------------------------------------------------- the 64-bit values ---
_C = {
    2: [(1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)],
    3: [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0),
        (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)],
}
_F64 = torch.float64


class _Method:
    """The penalized lattice step with rigid particles, 64 bits, any device."""

    def __init__(self, w, device):
        self.w, self.D, self.dev = w, w.D, device
        self.shape = (w.n[2], w.n[1], w.n[0])
        self.c = _C[w.D]
        self.Q = len(self.c)
        axis_w, edge_w, self.w0 = (1 / 9, 1 / 36, 4 / 9) if w.D == 2 else (1 / 18, 1 / 36, 1 / 3)
        self.wt = [axis_w if sum(map(abs, c)) == 1 else edge_w for c in self.c]
        self.opp = [self.c.index(tuple(-k for k in c)) for c in self.c]
        self.walls = [not w.periodic[d] for d in range(w.D)]
        t = lambda a: torch.tensor(np.asarray(a, np.float64), dtype=_F64, device=device)
        self.g, self.drive = t(w.g_grav[:w.D]), t(w.g_drive[:w.D])
        self.gmag = float(np.linalg.norm(w.g_grav))
        self.R = t(w.radius)
        self.Bm = t(w.minor) if getattr(w, "minor", None) is not None else None
        # per population: nodes whose source lies beyond a wall, and the moving-wall term there
        self.out, self.term = [], []
        for q, c in enumerate(self.c):
            m = torch.zeros(self.shape, dtype=torch.bool, device=device)
            tm = torch.zeros(self.shape, dtype=_F64, device=device) if w.wall_u is not None else None
            for d in range(w.D):
                if self.walls[d] and c[d]:
                    sl = [slice(None)] * 3
                    sl[2 - d] = 0 if c[d] > 0 else w.n[d] - 1
                    m[tuple(sl)] = True
                    if tm is not None:
                        uw = w.wall_u[d][0 if c[d] > 0 else 1]
                        tm[tuple(sl)] = 6.0 * self.wt[q] * sum(c[e] * uw[e] for e in range(3))
            self.out.append(m)
            self.term.append(tm)
        H = int(math.ceil(max(w.radius))) + 2 if w.radius else 1
        r = torch.arange(-H, H + 1, device=device)
        self.off = torch.stack(torch.meshgrid(*([r] * w.D), indexing="ij"), -1).reshape(-1, w.D)

    def start(self):
        z = lambda *s: torch.zeros(s, dtype=_F64, device=self.dev)
        P, nw = len(self.w.radius), 1 if self.D == 2 else 3
        X = torch.tensor(np.asarray(self.w.pos), dtype=_F64, device=self.dev).reshape(P, self.D)
        T = z(P, nw)
        if self.Bm is not None and self.w.theta is not None:
            T[:, 0] = torch.tensor(self.w.theta, dtype=_F64, device=self.dev)
        return z(self.Q, *self.shape), X, z(P, self.D), z(P, nw), T, z(P, self.D)

    def ratio(self):
        return torch.tensor(np.asarray(self.w.ratio), dtype=_F64, device=self.dev)

    def solid(self, X, T):
        """(particle, flat node, node coordinates relative to X's image) of every owned node."""
        n = torch.tensor(self.w.n[:self.D], device=self.dev)
        X = X.detach()
        node = torch.floor(X).long()[:, None, :] + self.off[None]
        r = node.to(_F64) - X[:, None, :]
        if self.Bm is None:
            inside = (r * r).sum(-1) <= (self.R * self.R)[:, None]
        else:
            co, si = torch.cos(T.detach()[:, :1]), torch.sin(T.detach()[:, :1])
            u, v = r[..., 0] * co + r[..., 1] * si, r[..., 1] * co - r[..., 0] * si
            a2, b2 = (self.R * self.R)[:, None], (self.Bm * self.Bm)[:, None]
            inside = b2 * u * u + a2 * v * v <= a2 * b2
        for d in range(self.D):
            if self.walls[d]:
                inside = inside & (node[..., d] >= 0) & (node[..., d] < n[d])
        wrapped = node % n
        flat = wrapped[..., 0] + self.w.n[0] * wrapped[..., 1]
        if self.D == 3:
            flat = flat + self.w.n[0] * self.w.n[1] * wrapped[..., 2]
        p, k = torch.nonzero(inside, as_tuple=True)
        flat, node = flat[p, k], node[p, k]
        owner = torch.full((math.prod(self.shape),), X.shape[0], dtype=torch.long, device=self.dev)
        owner.scatter_reduce_(0, flat, p, "amin")
        own = owner[flat] == p
        return p[own], flat[own], node[own].to(_F64)

    def stream(self, f):
        out = []
        for q, c in enumerate(self.c):
            v = torch.roll(f[q], (c[2], c[1], c[0]), (0, 1, 2))
            b = f[self.opp[q]] if self.term[q] is None else f[self.opp[q]] + self.term[q]
            out.append(torch.where(self.out[q], b, v))
        return out

    def moments(self, f, a):
        """u and p (Eq. 15); a: acceleration per axis (numbers or tensors)."""
        u = []
        for d in range(self.D):
            m = sum((f[q] if c[d] > 0 else -f[q]) for q, c in enumerate(self.c) if c[d])
            u.append(m + 0.5 * a[d])
        uu = sum(v * v for v in u)
        p = (sum(f) / 3.0 - 0.5 * self.w0 * uu) / (1.0 - self.w0)
        return u, uu, p

    def collide(self, f, a, u, uu, p, alpha=None):
        tau = self.w.tau
        base = p - 0.5 * uu
        ua = sum(v * w for v, w in zip(u, a))
        feq, F = [], []
        for q, c in enumerate(self.c):
            cu = sum(c[d] * u[d] for d in range(self.D) if c[d])
            ca = sum(c[d] * a[d] for d in range(self.D) if c[d])
            feq.append(3.0 * self.wt[q] * (base + cu + 1.5 * cu * cu))
            F.append((1.0 - 0.5 / tau) * 3.0 * self.wt[q] * (ca * (1.0 + 3.0 * cu) - ua))
        out = [f[q] - (f[q] - feq[q]) / tau + F[q] for q in range(self.Q)]
        if alpha is not None:
            D = self.D
            Pi = [[sum(c[i] * c[j] * (f[q] - feq[q]) for q, c in enumerate(self.c) if c[i] * c[j]) for j in range(D)]
                  for i in range(D)]
            tr = sum(Pi[i][i] for i in range(D)) / 3.0
            for q, c in enumerate(self.c):
                cc = sum(c[i] * c[j] * Pi[i][j] for i in range(D) for j in range(D) if c[i] * c[j])
                out[q] = out[q] + 4.5 * self.wt[q] * alpha * (cc - tr)
        return out

    def extent(self, T, d):
        if self.Bm is None:
            return self.R
        co, si = torch.cos(T[:, 0]), torch.sin(T[:, 0])
        e, ep = (co, si) if d == 0 else (si, co)
        return torch.sqrt((self.R * e) ** 2 + (self.Bm * ep) ** 2)

    def force(self, Y, T, Cc):
        """Pair and wall forces (Eqs. 19-21) at positions Y."""
        w, P = self.w, Y.shape[0]
        F = torch.zeros_like(Y)
        if P > 1:
            dd = Y[:, None] - Y[None]
            for d in range(self.D):
                if not self.walls[d]:
                    k = torch.round(dd[..., d].detach() / w.n[d]) * w.n[d]
                    dd = dd - k[..., None] * torch.nn.functional.one_hot(torch.tensor(d, device=self.dev), self.D)
            dist = torch.sqrt((dd * dd).sum(-1) + torch.eye(P, dtype=_F64, device=self.dev))
            sc = torch.clamp((self.R[:, None] + self.R[None] + w.delta - dist) / w.delta, min=0.0)
            F = F + (Cc / w.eps_p)[:, None] * (dd * (sc * sc)[..., None]).sum(1)
        cols = []
        for d in range(self.D):
            col = torch.zeros_like(Y[:, d])
            if self.walls[d]:
                for plane in (-0.5, w.n[d] - 0.5):
                    diff = 2.0 * (Y[:, d] - plane)
                    sc = torch.clamp((2.0 * self.extent(T, d) + w.delta - diff.abs()) / w.delta, min=0.0)
                    col = col + Cc / w.eps_w * diff * sc * sc
            cols.append(col)
        return F + torch.stack(cols, 1)

    def step(self, f, X, U, Wv, T, A, ratio, alpha):
        w, D, P = self.w, self.D, X.shape[0]
        p, flat, node = self.solid(X, T)
        fs = self.stream(f)
        drive = [float(v) for v in w.g_drive[:D]]
        u, uu, pr = self.moments(fs, drive)
        new = torch.stack(self.collide(fs, drive, u, uu, pr)).reshape(self.Q, -1)
        # the solid nodes: local acceleration, penalty, projection sums
        a_p = (1.0 - 1.0 / ratio)[:, None] * self.g + A + self.drive
        a = [a_p[p, d] for d in range(D)]
        fl = [v.reshape(-1)[flat] for v in fs]
        us, uus, ps = self.moments(fl, a)
        new = new.index_copy(1, flat, torch.stack(self.collide(fl, a, us, uus, ps, alpha))).reshape(self.Q, *self.shape)
        us, r = torch.stack(us, 1), node - X[p]
        z = lambda *s: torch.zeros(s, dtype=_F64, device=self.dev)
        cnt = z(P).index_add(0, p, torch.ones_like(flat, dtype=_F64))
        Un = z(P, D).index_add(0, p, us) / cnt[:, None]
        if D == 2:
            Lz = z(P).index_add(0, p, r[:, 0] * us[:, 1] - r[:, 1] * us[:, 0])
            Wn = (Lz / z(P).index_add(0, p, (r * r).sum(1)))[:, None]
        else:
            Lv = z(P, 3).index_add(0, p, torch.linalg.cross(r, us))
            eye = torch.eye(3, dtype=_F64, device=self.dev)
            I = z(P, 3, 3).index_add(0, p, (r * r).sum(1)[:, None, None] * eye - r[:, :, None] * r[:, None, :])
            Wn = torch.linalg.solve(I, Lv)
        # Algorithm 1
        h, Ub = 1.0 / w.K, 0.5 * (Un + U)
        Cc = (ratio - 1.0) * self.gmag
        Y, cor = X, torch.zeros_like(X)
        for _ in range(w.K):
            Ys = Y + h * Ub
            k = (0.25 * h * h / (ratio * cnt))[:, None] * (self.force(Y, T, Cc) + self.force(Ys, T, Cc))
            Y, cor = Ys + k, cor + k
        for d in range(D):
            if not self.walls[d]:
                n = w.n[d]
                wrap = torch.where(Y[:, d] >= n, -float(n), 0.0) + torch.where(Y[:, d] < 0, float(n), 0.0)
                Y = Y + wrap.detach()[:, None] * torch.nn.functional.one_hot(torch.tensor(d, device=self.dev), D)
        return new, Y, Un, Wn, T + 0.5 * (Wn + Wv), 2.0 * cor, cnt

    def fields(self, f, X, T, A, ratio):
        """u [D, ...] and p of the state, as the next step sees it."""
        p, flat, _ = self.solid(X, T)
        fs = self.stream(f)
        a = [torch.full((math.prod(self.shape),), float(v), dtype=_F64, device=self.dev) for v in self.w.g_drive[:self.D]]
        a_p = (1.0 - 1.0 / ratio)[:, None] * self.g + A
        for d in range(self.D):
            a[d] = a[d].index_add(0, flat, a_p[p, d])
        u, _, pr = self.moments([v.reshape(-1) for v in fs], a)
        return torch.cat(u), pr


def _run_exact(w, steps, device, every=0):
    """State after `steps` steps, and with `every` the particle states on the way."""
    m = _Method(w, device)
    f, X, U, Wv, T, A = m.start()
    ratio, frames, cnt = m.ratio(), [], None
    with torch.no_grad():
        for k in range(steps):
            f, X, U, Wv, T, A, cnt = m.step(f, X, U, Wv, T, A, ratio, w.alpha)
            if every and (k + 1) % every == 0:
                frames.append((X, U, Wv, T, A))
        if every:
            return frames
        return m.fields(f, X, T, A, ratio), (X, U, Wv, T, A)


def _exact_gradient(case, seed, device):
    D = 3 if case["nz"] > 1 else 2
    al, ra, X0, U0, gX, gU = (torch.from_numpy(a).to(device, _F64) for a in _gradient_inputs(case, seed))
    outs = {k: [] for k in ("X", "U", "alpha", "ratio", "X0", "U0")}
    for b in range(case["batch"]):
        w = W.Workload("gradient", D, (case["nx"], case["ny"], case["nz"]), (0, 0, 1 if D == 2 else 0), 1.0, 1.0,
                       g_grav=_gravity(D), pos=X0[b].tolist(), radius=[case["radius"]] * case["np"], ratio=ra[b].tolist())
        m = _Method(w, device)
        leaves = [t.clone().requires_grad_(True) for t in (al[b], ra[b], X0[b], U0[b])]
        a, r, X, U = leaves
        f, _, _, Wv, T, A = m.start()
        for _ in range(case["steps"]):
            f, X, U, Wv, T, A, _ = torch.utils.checkpoint.checkpoint(m.step, f, X, U, Wv, T, A, r, a, use_reentrant=False)
        g = torch.autograd.grad((X, U), leaves, (gX[b], gU[b]))
        for k, v in zip(outs, (X.detach(), U.detach(), *g)):
            outs[k].append(v)
    return {k: torch.stack(v) for k, v in outs.items()}


def _exact_projection(case, seed, device):
    w = _scene(case, seed)[0]
    m, D, P = _Method(w, device), w.D, w.num_particles
    _, X, _, _, T, _ = m.start()
    p, flat, node = m.solid(X, T)
    us = _velocity(w.n, D, seed).reshape(D, -1)[:, flat].to(_F64).T
    r = node - X[p]
    z = lambda *s: torch.zeros(s, dtype=_F64, device=device)
    cnt = z(P).index_add(0, p, torch.ones_like(flat, dtype=_F64))
    vel = z(P, D).index_add(0, p, us) / cnt[:, None]
    if D == 2:
        om = z(P).index_add(0, p, r[:, 0] * us[:, 1] - r[:, 1] * us[:, 0]) / z(P).index_add(0, p, (r * r).sum(1))
        om = om[:, None]
    else:
        eye = torch.eye(3, dtype=_F64, device=device)
        I = z(P, 3, 3).index_add(0, p, (r * r).sum(1)[:, None, None] * eye - r[:, :, None] * r[:, None, :])
        om = torch.linalg.solve(I, z(P, 3).index_add(0, p, torch.linalg.cross(r, us)))
    return {"vel": vel, "omega": om, "count": None}


def exact(case, seed, device="cuda"):
    out = _exact(case, seed, device)
    if out is not None and case["kind"] not in ("gradient", "projection"):
        # no value: the spin of spheres that settle from rest without touching (rounding alone
        # turns them), and what 16-bit populations do not resolve, the same spin in 2D and the
        # pressure of a nearly uniform flow
        none = ("W", "theta") if case["scene"] == "spheres" else ()
        none = ("p", "W", "theta") if case["storage"] == "fp16" else none
        out.update({k: None for k in none if k in out})
    return out


def _exact(case, seed, device):
    kind = case["kind"]
    if kind == "projection":
        return _exact_projection(case, seed, device)
    if kind == "gradient":
        # about four forward steps' time per step and node, D3Q19 2.5 times as much
        n = 4 * case["batch"] * case["nx"] * case["ny"] * case["nz"] * case["steps"] * (2.5 if case["nz"] > 1 else 1)
        return _exact_gradient(case, seed, device) if n <= _EXACT_NODE_STEPS else None
    ws = _scene(case, seed)
    steps = case["frames"] * case["every"] if kind == "frames" else case["steps"]
    if sum(w.nodes for w in ws) * steps * (2.5 if ws[0].D == 3 else 1.0) > _EXACT_NODE_STEPS:
        return None
    if kind == "frames":
        frames = _run_exact(ws[0], steps, device, every=case["every"])
        D, out = ws[0].D, {}
        for k, name in enumerate(("X", "U", "W", "theta", "A")):
            v = torch.stack([fr[k] for fr in frames])
            full = torch.zeros((*v.shape[:2], 3), dtype=_F64, device=device)
            if v.shape[2] == 1:
                full[:, :, 2] = v[:, :, 0]
            else:
                full[:, :, :v.shape[2]] = v
            out[name] = full
        return {**out, "count": None}
    us, ps, parts = [], [], []
    for w in ws:
        (u, p), part = _run_exact(w, steps, device)
        us.append(u)
        ps.append(p)
        parts.append(part)
    out = {"u": torch.cat(us), "p": torch.cat(ps), "owner": None}
    if kind == "job":
        for k, name in enumerate(("X", "U", "W", "theta", "A")):
            out[name] = torch.cat([q[k] for q in parts])
        out["count"] = None
    return out
