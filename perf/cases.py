"""The measured workloads of this library, each one pass through the public entry points.

A case is a plain dict; ``prepare`` makes what a program has in hand before the call (the
simulation handle and its initial state on the GPU), ``run`` is one pass, ``work`` what the
pass cannot do without, and ``exact`` the same pass in 64 bits in plain torch.

Kinds of case:
  sim      advance one simulation by ``steps`` time steps, ``parts`` times, and read the
           moments after each part and the raw state at the end (a solver's output interval);
  batch    advance many uneven 2D channels together and read every instance's moments;
  rollout  differentiable rollout: forward with checkpoints, then the adjoint sweep for the
           gradients of the force field, the wall velocities and the initial state;
  graded   the non-uniform (tanh) mesh, with the steady-state residual at the end;
  monitor  the diagnostics of a running simulation: FP64 residual and totals, and the moments.
"""
import math

import numpy as np
import torch

from paper_1411_6121_gb300 import autograd, dugks
from paper_1411_6121_gb300 import workloads as W

STORES = {"f32": dugks.STORE_F32, "bf16": dugks.STORE_BF16, "f16": dugks.STORE_F16, "f64": dugks.STORE_F64}
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16, "f64": torch.float64}
BYTES = {"f32": 4, "bf16": 2, "f16": 2, "f64": 8}
F16_SCALE = 4096.0  # F16 storage holds g~ * 2^12
# floating-point operations of one cell update (step 1, interfaces, update), per velocity set
FLOPS = {9: 450, 19: 1500, 27: 2600}


def listed():
    return [
        # the smallest use: a channel driven to its steady state, 1,000 steps between looks at it;
        # 256 cells, so a step is all latency
        dict(name="channel_8x32", kind="sim", q=9, nx=8, ny=32, nz=1, store="f32", flow="channel", steps=1000, parts=1),
        # oscillating channel (Womersley): the moments at four phases of a run
        dict(name="womersley_128x64", kind="sim", q=9, nx=128, ny=64, nz=1, store="f32", flow="womersley", steps=250,
             parts=4),
        # the 2D lid-driven cavity at its benchmark size
        dict(name="cavity_1024", kind="sim", q=9, nx=1024, ny=1024, nz=1, store="f32", flow="cavity", steps=100, parts=1),
        # 16-bit storage, pressure inlet and outlet between bounce-back walls, sizes that fit no tile
        dict(name="duct_1277x611_f16", kind="sim", q=9, nx=1277, ny=611, nz=1, store="f16", flow="duct", steps=100,
             parts=1),
        # the 3D cube at the size of a parameter study
        dict(name="cube_64", kind="sim", q=19, nx=64, ny=64, nz=64, store="f32", flow="cavity", steps=100, parts=1),
        # the 3D cube at the benchmark's size, FP32 and 16-bit storage
        dict(name="cube_256", kind="sim", q=19, nx=256, ny=256, nz=256, store="f32", flow="cavity", steps=10, parts=1),
        dict(name="cube_256_bf16", kind="sim", q=19, nx=256, ny=256, nz=256, store="bf16", flow="cavity", steps=10,
             parts=1),
        # the full 3D velocity set, a channel driven by a per-cell force field, ragged sizes
        dict(name="channel27_157x101x83", kind="sim", q=27, nx=157, ny=101, nz=83, store="f32", flow="forced", steps=20,
             parts=1),
        # many uneven channels advanced together (a parameter sweep)
        dict(name="batch_64", kind="batch", count=64, specs=0x1411, steps=200),
        # gradients of a rollout on the largest of those channels
        dict(name="rollout_512x256", kind="rollout", nx=512, ny=256, steps=200, every=50),
        # the graded cavity in FP64 with its steady-state residual
        dict(name="graded_128_f64", kind="graded", nx=128, ny=128, store="f64", steps=200),
        # residual, totals and moments of the 256^3 cube
        dict(name="monitor_256", kind="monitor", q=19, nx=256, ny=256, nz=256, store="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(rng, cells, lo, hi, store):
    # BF16 in short intervals: its storage noise grows with the steps (half a percent of the
    # state after some tens) and would hide everything else
    return max(lo, min(hi if store != "bf16" else 20, int(rng.uniform(0.5, 1.0) * 1e8 / cells)))


def draw(rng):
    kind = rng.choice(["sim2d", "sim2d", "sim2d", "sim19", "sim19", "sim27", "batch", "rollout", "graded", "monitor"])
    if kind == "sim2d":
        nx, ny = _log_int(rng, 8, 1500), _log_int(rng, 8, 1000)
        store, parts = rng.choice(["f32", "f32", "f16", "bf16"]), rng.choice([1, 1, 4])
        if store != "f32":
            parts = 1
        return dict(kind="sim", q=9, nx=nx, ny=ny, nz=1, store=store,
                    flow=rng.choice(["channel", "womersley", "cavity", "duct", "forced"]),
                    steps=_steps(rng, nx * ny, 20, 1000 // parts, store), parts=parts)
    if kind in ("sim19", "sim27"):
        q, top = (19, 220) if kind == "sim19" else (27, 150)
        nx, ny, nz = (_log_int(rng, 12, top) for _ in range(3))
        store = rng.choice(["f32", "f32", "f16", "bf16"])
        return dict(kind="sim", q=q, nx=nx, ny=ny, nz=nz, store=store,
                    flow=rng.choice(["channel", "cavity", "duct", "forced"]),
                    steps=_steps(rng, nx * ny * nz, 8, 150, store), parts=1)
    if kind == "batch":
        return dict(kind="batch", count=_log_int(rng, 4, 64), specs=rng.randrange(1 << 16), steps=rng.randrange(20, 201))
    if kind == "rollout":
        nx, ny = _log_int(rng, 16, 600), _log_int(rng, 16, 300)
        return dict(kind="rollout", nx=nx, ny=ny, steps=rng.randrange(60, 201), every=rng.choice([20, 50, 100]))
    if kind == "graded":
        return dict(kind="graded", nx=_log_int(rng, 24, 200), ny=_log_int(rng, 24, 200),
                    store=rng.choice(["f32", "f64"]), steps=rng.randrange(50, 201))
    q = rng.choice([9, 19, 27])
    top = {9: 2000, 19: 240, 27: 200}[q]
    return dict(kind="monitor", q=q, nx=_log_int(rng, 16, top), ny=_log_int(rng, 16, top),
                nz=_log_int(rng, 16, top) if q > 9 else 1, store=rng.choice(["f32", "f16", "bf16"]))


# ---- inputs -----------------------------------------------------------------------

def _shape(case):
    return (case["nx"], case["ny"]) if case.get("nz", 1) == 1 and case.get("q", 9) == 9 else \
        (case["nx"], case["ny"], case["nz"])


def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _lattice(q):
    if q == 9:
        e = [(a, b, 0) for a in (-1, 0, 1) for b in (-1, 0, 1)]
        w = [(1 / 6, 2 / 3, 1 / 6)[a + 1] * (1 / 6, 2 / 3, 1 / 6)[b + 1] for a, b, _ in e]
        return e, w
    e = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
    if q == 27:
        return e, [math.prod((1 / 6, 2 / 3, 1 / 6)[x + 1] for x in v) for v in e]
    e = [v for v in e if abs(v[0]) + abs(v[1]) + abs(v[2]) < 3]
    return e, [(1 / 3, 1 / 18, 1 / 36)[abs(v[0]) + abs(v[1]) + abs(v[2])] for v in e]


def _fields(shape, gen, u_amp=0.03, p_amp=1e-3):
    """Smooth velocity modes with random phases plus cell noise, and pressure noise, FP64 on the
    GPU, cells x fastest: p [...], u [dim][...] with the tensor axes (z,) y, x."""
    dim = len(shape)
    dims = tuple(reversed(shape))
    ph = (torch.rand((dim, dim), generator=gen, device="cuda", dtype=torch.float64) * 2 * math.pi).cpu()
    u = []
    for a in range(dim):
        f = torch.full((1,) * dim, 0.8 * u_amp, dtype=torch.float64, device="cuda")
        for b in range(dim):
            x = (torch.arange(shape[b], device="cuda", dtype=torch.float64) + 0.5) / shape[b]
            f = f * torch.sin(2 * math.pi * x + ph[a, b].item()).reshape([-1 if d == dim - 1 - b else 1 for d in range(dim)])
        u.append(f + 0.1 * u_amp * torch.randn(dims, generator=gen, device="cuda", dtype=torch.float32).double())
    p = p_amp * torch.randn(dims, generator=gen, device="cuda", dtype=torch.float32).double()
    return p, u


def _equilibrium(q, p, u, store):
    """The initial state of Sec. 3, f_eq(rho0 + p/RT, u) - W rho0, in the storage type, [q][ncell]
    (lattice units: c = 1, rho0 = 1, RT = 1/3)."""
    e, w = _lattice(q)
    uu = sum(x * x for x in u)
    out = torch.empty((q, p.numel()), dtype=DTYPES[store], device="cuda")
    scale = F16_SCALE if store == "f16" else 1.0
    for k in range(q):
        eu = 0.0
        for a in range(len(u)):
            if e[k][a]:
                eu = eu + e[k][a] * u[a]
        g = w[k] * (3.0 * p + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu)
        out[k] = (g * scale).reshape(-1).to(out.dtype)
    return out


def _setup(case):
    """Flow parameters in lattice units (dx = 1, RT = 1/3, rho0 = 1, dt = 0.5)."""
    shape = _shape(case)
    dim, H = len(shape), case["ny"]
    flow = case["flow"]
    cfg = dict(shape=shape, q=case["q"], dt=W.dt_for(), rt=W.RT_LATTICE, rho0=W.RHO0)
    if flow == "channel":
        cfg.update(nu=0.01 if dim == 2 else 0.05, g=(1e-5 * min(1.0, 32 / H), 0.0, 0.0), bcs=W.channel_bcs(dim))
    elif flow == "womersley":
        nu = 0.2
        cfg.update(nu=nu, g=(1e-4 * min(1.0, 64 / H), 0.0, 0.0), omega=nu * (2.0 * 4.0 / H) ** 2, bcs=W.channel_bcs(dim))
    elif flow == "cavity":
        cfg.update(nu=max(0.1 * case["nx"] / 1000.0, 0.005), bcs=W.cavity_bcs(dim, 0.1))
    elif flow == "duct":
        p = 1e-3 * min(1.0, 64 / H)
        cfg.update(nu=0.1, bcs=[W.pressure(p), W.pressure(-p), W.bounce_back(), W.bounce_back((0.01, 0.0, 0.0))] +
                   ([W.periodic()] * 2 if dim == 3 else []))
    else:  # forced: a channel under a per-cell acceleration field
        cfg.update(nu=0.05, bcs=W.channel_bcs(dim))
    return cfg


def _force_field(shape, gen, G):
    n = math.prod(shape)
    f = torch.zeros((len(shape), n), dtype=torch.float32, device="cuda")
    f[0] = G * (1.0 + 0.1 * torch.randn(n, generator=gen, device="cuda"))
    return f


def _sim_inputs(case, seed):
    gen = _gen(seed)
    shape = _shape(case)
    state0 = _equilibrium(case["q"], *_fields(shape, gen), case["store"])
    field = None
    if case.get("flow") == "forced":
        field = _force_field(shape, gen, 8.0 * 0.05 * 0.05 / case["ny"] ** 2)
    return state0, field


def _batch_inputs(case, seed):
    ins, init = [], []
    for i, sp in enumerate(W.batched_channels(case["count"], seed=case["specs"])):
        gen = _gen(seed, i + 1)
        p, u = _fields(sp["shape"], gen, u_amp=0.02, p_amp=1e-4)
        ins.append(dict(shape=sp["shape"], nu=sp["nu"], bcs=sp["bcs"], field=_force_field(sp["shape"], gen, sp["g"][0])))
        init.append((p, torch.stack(u)))
    return ins, init


def _rollout_inputs(case, seed):
    gen = _gen(seed)
    shape = (case["nx"], case["ny"])
    n, H = math.prod(shape), case["ny"]
    nu = 0.05
    state0 = _equilibrium(9, *_fields(shape, gen), "f32")
    field = _force_field(shape, gen, 8.0 * nu * 0.05 / H ** 2)
    wall = torch.zeros((6, 3), dtype=torch.float32)
    wall[3, 0] = 0.01
    dmom = torch.randn((3, n), generator=gen, device="cuda", dtype=torch.float32) / n
    return nu, state0, field, wall, dmom


def _graded_cfg(case):
    shape = (case["nx"], case["ny"])
    faces = [W.tanh_faces(n, length=float(n)) for n in shape]
    dt = 0.5 * min(float(np.diff(f).min()) for f in faces)
    return dict(shape=shape, q=9, nu=0.1 * case["nx"] / 400.0, dt=dt, bcs=W.cavity_bcs(2, 0.1), faces=faces)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sim":
        state0, field = _sim_inputs(case, seed)
        sim = dugks.Sim(field=field, store=STORES[case["store"]], **_setup(case))
        torch.cuda.synchronize()
        sim.set_state(state0)
        moms = [torch.empty((sim.dim + 1, sim.ncell), dtype=torch.float32, device="cuda") for _ in range(case["parts"])]
        # 16-bit states: the state alone (the stored values are what the rounding acts on)
        return dict(case=case, sim=sim, state=state0, moms=moms if case["store"] == "f32" else [None] * case["parts"])
    if kind == "batch":
        ins, init = _batch_inputs(case, seed)
        b = dugks.Batch(ins, dt=W.dt_for())
        b.tune()
        for i, (p, u) in enumerate(init):
            b.init(i, p=p.cpu().numpy(), u=u.cpu().numpy())
        return dict(case=case, batch=b)
    if kind == "rollout":
        nu, state0, field, wall, dmom = _rollout_inputs(case, seed)
        sim = dugks.Sim(shape=(case["nx"], case["ny"]), q=9, nu=nu, dt=W.dt_for(), bcs=W.channel_bcs(2), field=field)
        for t in (field, wall, state0):
            t.requires_grad_(True)
        return dict(case=case, sim=sim, state=state0, field=field, wall=wall, dmom=dmom)
    if kind == "graded":
        gen = _gen(seed)
        state0 = _equilibrium(9, *_fields((case["nx"], case["ny"]), gen), case["store"])
        sim = dugks.Sim(store=STORES[case["store"]], **_graded_cfg(case))
        torch.cuda.synchronize()
        sim.set_state(state0)
        sim.residual()
        return dict(case=case, sim=sim, state=state0)
    shape = _shape(case)  # monitor: the velocity of one state kept by the first residual, then another state
    first, second = (_equilibrium(case["q"], *_fields(shape, _gen(seed, s)), case["store"]) for s in (1, 2))
    sim = dugks.Sim(shape=shape, q=case["q"], nu=0.05, dt=W.dt_for(), bcs=W.cavity_bcs(len(shape), 0.1),
                    store=STORES[case["store"]])
    torch.cuda.synchronize()
    sim.set_state(first)
    sim.residual()
    sim.set_state(second)
    return dict(case=case, sim=sim, mom=torch.empty((sim.dim + 1, sim.ncell), dtype=torch.float32, device="cuda"))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "sim":
        out = {}
        for i, mom in enumerate(s["moms"]):
            s["sim"].step(case["steps"])
            if mom is not None:
                out["moments%d" % i] = s["sim"].moments(mom)
        out["state"] = s["sim"].get_state(s["state"])
        return out
    if kind == "batch":
        s["batch"].step(case["steps"])
        return [s["batch"].moments(i) for i in range(case["count"])]
    if kind == "rollout":
        mom = autograd.rollout(s["sim"], s["field"], s["wall"], case["steps"], every=case["every"], state0=s["state"])
        df, dw, ds = torch.autograd.grad(mom, (s["field"], s["wall"], s["state"]), s["dmom"])
        return {"moments": mom.detach(), "dfield": df, "dwall": dw, "dstate": ds}
    if kind == "graded":
        s["sim"].step(case["steps"])
        r = s["sim"].residual()
        # FP32 storage: the residual in the precision of the state it measures
        return {"state": s["sim"].get_state(s["state"]), "residual": r if case["store"] == "f64" else r.astype(np.float32)}
    return {"residual": s["sim"].residual(), "moments": s["sim"].moments(s["mom"])}


def work(case):
    """Per step: the state read and written once (and the force field read); the moments and the
    raw state handed out once per pass. The adjoint's reverse step: the state, lambda in and out,
    the field and its gradient, and the forward recompute."""
    kind = case["kind"]
    if kind == "batch":
        specs = W.batched_channels(case["count"], seed=case["specs"])
        n = sum(math.prod(s["shape"]) for s in specs)
        return {"bytes": n * (case["steps"] * (72 + 8) + 48), "flops": n * case["steps"] * FLOPS[9]}
    if kind == "rollout":
        n, T = case["nx"] * case["ny"], case["steps"]
        return {"bytes": n * T * (80 + 80 + 132), "flops": n * T * 4 * FLOPS[9]}
    q = case.get("q", 9)
    n = math.prod(_shape(case) if "nz" in case else (case["nx"], case["ny"]))
    state, mom = q * BYTES[case["store"]], 4 * (3 if q == 9 else 4)
    if kind == "monitor":
        dim = 2 if q == 9 else 3
        return {"bytes": n * (2 * state + mom + 2 * 8 * dim), "flops": n * 2 * 4 * q}
    steps = case["steps"] * case.get("parts", 1)
    field = 4 * len(_shape(case)) if case.get("flow") == "forced" else 0
    return {"bytes": n * (steps * (2 * state + field) + 2 * state + (mom if case["store"] == "f32" else 0)),
            "flops": n * steps * FLOPS[q]}


# ---- the same passes in 64 bits -----------------------------------------------------

class _Scheme:
    """The scheme (Appendix steps 1-10) on tensors [q][(z)][y][x] of the deviation f~ - W rho0, in
    FP64, all velocities at once; uniform meshes are graded ones with equal widths."""

    def __init__(self, shape, q, nu, dt, bcs, rt=1.0 / 3.0, rho0=1.0, g=(0.0, 0.0, 0.0), omega=0.0, faces=None, field=None):
        self.D, self.shape, self.q, self.dt, self.rt, self.rho0, self.omega = len(shape), shape, q, dt, rt, rho0, omega
        self.c, self.h, self.tau = math.sqrt(3.0 * rt), 0.5 * dt, nu / rt
        e, w = _lattice(q)
        one = (q,) + (1,) * self.D
        self.e = [torch.tensor([float(v[a]) for v in e], dtype=torch.float64, device="cuda").reshape(one) for a in range(self.D)]
        self.w = torch.tensor(w, dtype=torch.float64, device="cuda").reshape(one)
        self.opp = torch.tensor([e.index((-v[0], -v[1], -v[2])) for v in e], device="cuda")
        self.bcs = [tuple(b) + (0.0,) * (4 - len(b)) for b in list(bcs) + [W.periodic()] * (6 - len(bcs))]
        self.wall = [[float(x) for x in b[1]] for b in self.bcs]
        self.g = g
        self.field = None if field is None else field.double().reshape((self.D,) + tuple(reversed(shape)))
        self.axes = []
        for a in range(self.D):
            n = shape[a]
            xf = torch.arange(n + 1, dtype=torch.float64) if faces is None else torch.as_tensor(faces[a], dtype=torch.float64)
            xc = 0.5 * (xf[1:] + xf[:-1])
            if self.per(a):
                lo, hi = xc[-1:] - (xf[-1] - xf[0]), xc[:1] + (xf[-1] - xf[0])
            else:
                lo, hi = 2 * xf[:1] - xc[:1], 2 * xf[-1:] - xc[-1:]
            x = torch.cat([lo, xc, hi])
            eg = [float((x[0] - x[1]) / (x[2] - x[1])), float((x[-1] - x[-2]) / (x[-3] - x[-2]))] if n > 1 else [0.0, 0.0]
            sh = [-1 if d == self.D - 1 - a else 1 for d in range(self.D)]
            self.axes.append(dict(w=((xf - x[:-1]) / (x[1:] - x[:-1])).cuda().reshape(sh),
                                  idc=(1.0 / (x[1:] - x[:-1])).cuda().reshape(sh),
                                  width=(xf[1:] - xf[:-1]).cuda().reshape(sh), eg=eg))

    def per(self, a):
        return self.bcs[2 * a][0] == W.BC_PERIODIC

    def cut(self, f, a, lo, hi):
        """Entries lo .. hi - 1 (from the end where not positive) along axis a."""
        dim = f.dim() - 1 - a
        n = f.shape[dim]
        return f.narrow(dim, lo, (hi if hi > 0 else n + hi) - lo)

    def at(self, f, a, i):
        dim = f.dim() - 1 - a
        return f.narrow(dim, i if i >= 0 else f.shape[dim] + i, 1)

    def accel(self, t):
        G = []
        for a in range(self.D):
            v = float(self.g[a]) * torch.ones((1,) * self.D, dtype=torch.float64, device="cuda")
            G.append((v if self.field is None else v + self.field[a]) * math.cos(self.omega * t))
        return G

    def moments(self, f, G, wt):
        """drho and m = rho0 u / c."""
        return f.sum(0), [(f * self.e[a]).sum(0) + self.rho0 * G[a] / self.c * wt for a in range(self.D)]

    def geq(self, drho, m):
        em = sum(self.e[a] * m[a] for a in range(self.D))
        mm = sum(x * x for x in m)
        return self.w * (drho + 3.0 * em + (4.5 * em * em - 1.5 * mm) / self.rho0)

    def relax(self, f, G, wt, b, c):
        drho, m = self.moments(f, G, wt)
        q = self.geq(drho, m)
        out = f + b * (q - f)
        if self.forced:
            s = 3.0 * sum((self.e[a] - m[a] / self.rho0) * (G[a] / self.c) for a in range(self.D))
            out = out + c * s * (self.w * self.rho0 + q)
        return out

    @property
    def forced(self):
        return self.field is not None or any(self.g)

    def face_G(self, G, d):
        out = []
        for x in G:
            if x.shape[x.dim() - 1 - d] == 1 and self.field is None:
                out.append(x)
                continue
            lo, hi = (self.at(x, d, -1), self.at(x, d, 0)) if self.per(d) else (self.at(x, d, 0), self.at(x, d, -1))
            x = torch.cat([lo, x, hi], x.dim() - 1 - d)
            L, R = self.cut(x, d, 0, -1), self.cut(x, d, 1, 0)
            out.append(L + self.axes[d]["w"] * (R - L))
        return out

    def sub(self, G, d, i):
        return [x if x.shape[x.dim() - 1 - d] == 1 else self.at(x, d, i) for x in G]

    def step(self, g, t, field=None, wall=None):
        if field is not None:
            self.field = field.double().reshape(self.field.shape)
        wall = self.wall if wall is None else wall.double().cuda()
        D, tau, dt, h = self.D, self.tau, self.dt, self.h
        fp = self.relax(g, self.accel(t), 0.5 * dt, 3 * h / (2 * tau + dt), 3 * tau * h / (2 * tau + dt))
        ext = fp
        for a in range(D):
            dim = ext.dim() - 1 - a
            if self.per(a):
                lo, hi = self.at(ext, a, -1), self.at(ext, a, 0)
            else:
                eg = self.axes[a]["eg"]
                lo = self.at(ext, a, 0) + eg[0] * (self.at(ext, a, 1) - self.at(ext, a, 0))
                hi = self.at(ext, a, -1) + eg[1] * (self.at(ext, a, -2) - self.at(ext, a, -1))
            ext = torch.cat([lo, ext, hi], dim)
        new = 4.0 / 3.0 * fp - g / 3.0
        Gh = self.accel(t + h)
        hc = h * self.c
        for d in range(D):
            ax = self.axes[d]
            band = ext  # cells around the interfaces, tangential axes trimmed
            for a in range(D):
                if a != d:
                    band = self.cut(band, a, 1, -1)
            L, R = self.cut(band, d, 0, -1), self.cut(band, d, 1, 0)
            F = L + ax["w"] * (R - L) - hc * self.e[d] * (R - L) * ax["idc"]
            for s in range(D):
                if s == d:
                    continue
                v = ext
                for a in range(D):
                    if a != d and a != s:
                        v = self.cut(v, a, 1, -1)
                Lv, Rv = self.cut(v, d, 0, -1), self.cut(v, d, 1, 0)
                v = Lv + ax["w"] * (Rv - Lv)
                lo, hi = self.cut(v, s, 0, -1), self.cut(v, s, 1, 0)
                v = lo + self.axes[s]["w"] * (hi - lo)  # cross points
                F = F - hc * self.e[s] * (self.cut(v, s, 1, 0) - self.cut(v, s, 0, -1)) / self.axes[s]["width"]
            Gf = self.face_G(Gh, d)
            if not self.per(d):
                ends = [self.wall_value(F, Gf, d, side, t, wall) for side in (0, 1)]
                F = torch.cat([ends[0], self.cut(F, d, 1, -1), ends[1]], F.dim() - 1 - d)
            f = self.relax(F, Gf, 0.5 * h, h / (2 * tau + h), tau * h / (2 * tau + h))
            new = new - dt * self.c * self.e[d] * (self.cut(f, d, 1, 0) - self.cut(f, d, 0, -1)) / ax["width"]
        return new

    def wall_value(self, F, Gf, d, side, t, wall):
        w = 2 * d + side
        kind, _, p, p_amp = self.bcs[w]
        Fw, Fc = self.at(F, d, 0 if side == 0 else -1), self.at(F, d, 1 if side == 0 else -2)
        mw = [wall[w][a] * (self.rho0 / self.c) for a in range(self.D)]
        if kind == W.BC_BOUNCE_BACK:
            new = Fw[self.opp] + 6.0 * self.w * sum(self.e[a] * mw[a] for a in range(self.D))
        else:
            drho, m = self.moments(Fc, self.sub(Gf, d, 1 if side == 0 else -2), 0.5 * self.h)
            if kind == W.BC_NEQ_VELOCITY:
                one = torch.ones_like(drho)
                qa = self.geq(drho, [x * one for x in mw])
            else:
                pw = p + p_amp * math.cos(self.omega * (t + self.h))
                qa = self.geq(torch.full_like(drho, pw / self.rt), m)
            new = qa + Fc - self.geq(drho, m)
        return torch.where(self.e[d] * (1.0 if side else -1.0) < 0, new, Fw)

    def out_moments(self, g, t):
        """[dim + 1][ncell]: p = drho RT, u."""
        drho, m = self.moments(g, self.accel(t), 0.5 * self.dt)
        return torch.stack([drho * self.rt] + [x * (self.c / self.rho0) for x in m]).reshape(self.D + 1, -1)

    def advance(self, g, n, first=0):
        for i in range(n):
            g = self.step(g, (first + i) * self.dt)
        return g

    def residual(self, g, before, t, t_before):
        u, v = self.out_moments(g, t)[1:], self.out_moments(before, t_before)[1:]
        rho = g.sum(0) + self.rho0
        return torch.cat([((u - v).norm() / u.norm()).reshape(1), rho.sum().reshape(1), self.rho0 * u.sum(1)])


def _shaped(state, shape, store):
    g = state.double().reshape((state.shape[0],) + tuple(reversed(shape)))
    return g / F16_SCALE if store == "f16" else g


def exact(case, seed):
    kind = case["kind"]
    if kind == "sim":
        shape = _shape(case)
        state0, field = _sim_inputs(case, seed)
        sch = _Scheme(field=field, **_setup(case))
        g, out = _shaped(state0, shape, case["store"]), {}
        del state0
        for i in range(case["parts"]):
            g = sch.advance(g, case["steps"], i * case["steps"])
            if case["store"] == "f32":
                out["moments%d" % i] = sch.out_moments(g, (i + 1) * case["steps"] * sch.dt)
        out["state"] = g.reshape(case["q"], -1) * (F16_SCALE if case["store"] == "f16" else 1.0)
        return out
    if kind == "batch":
        res = []
        for ins, (p, u) in zip(*_batch_inputs(case, seed)):
            sch = _Scheme(ins["shape"], 9, ins["nu"], W.dt_for(), ins["bcs"], field=ins["field"])
            g = _equilibrium(9, p, list(u), "f64").reshape((9,) + tuple(reversed(ins["shape"])))
            res.append(sch.out_moments(sch.advance(g.float().double(), case["steps"]), case["steps"] * sch.dt))
        return res
    if kind == "rollout":
        from torch.utils.checkpoint import checkpoint
        nu, state0, field, wall, dmom = _rollout_inputs(case, seed)
        shape = (case["nx"], case["ny"])
        sch = _Scheme(shape, 9, nu, W.dt_for(), W.channel_bcs(2), field=field)
        state, field, wall = (x.double().requires_grad_(True) for x in (state0, field, wall))
        g = _shaped(state, shape, "f32")
        for i in range(case["steps"]):
            g = checkpoint(sch.step, g, i * sch.dt, field, wall, use_reentrant=False)
        sch.field = field.reshape(sch.field.shape)
        mom = sch.out_moments(g, case["steps"] * sch.dt)
        df, dw, ds = torch.autograd.grad(mom, (field, wall, state), dmom.double())
        return {"moments": mom.detach(), "dfield": df, "dwall": dw, "dstate": ds}
    if kind == "graded":
        shape = (case["nx"], case["ny"])
        sch = _Scheme(**_graded_cfg(case))
        g0 = _shaped(_equilibrium(9, *_fields(shape, _gen(seed)), case["store"]), shape, case["store"])
        g = sch.advance(g0, case["steps"])
        return {"state": g.reshape(9, -1), "residual": sch.residual(g, g0, 0.0, 0.0)}
    shape = _shape(case)
    sch = _Scheme(shape, case["q"], 0.05, W.dt_for(), W.cavity_bcs(len(shape), 0.1))
    first, second = (_shaped(_equilibrium(case["q"], *_fields(shape, _gen(seed, s)), case["store"]), shape, case["store"])
                     for s in (1, 2))
    return {"residual": sch.residual(second, first, 0.0, 0.0), "moments": sch.out_moments(second, 0.0)}
