"""What the performance of this framework is measured on.

Each case is a piece of work that a user's program has the library do, through
the public binding (`ugkwp.Simulation`, `ugkwp.Batch`): time steps of a running
case in both precisions and at both orders, a whole short run, a batch, the
gas-kinetic start-up, the adjoint, reading the fields, and a restart from a
checkpoint.  Sizes, gas parameters and options are those of the workloads,
tests and benchmark of this repository.

A running case is entered through a state image, as a program that restarts
from a checkpoint does: each cell holds the particle population that the
method settles at (sampling balanced by collisions), with Maxwellian
velocities, uniform positions and a wave part for the rest, all drawn from the
seed.
"""
import functools
import math

import numpy as np
import torch

from paper_2007_13091_gb300 import ugkwp, workloads as wl

STEP = 1000  # step counter of the images (particles were born in earlier steps)


def listed():
    return [
        # the smallest calls: one small tube of the batch's range, two steps at
        # a time with the fields read after each; launches and latency count
        dict(name="steps_tube_2k_mixed_o1", kind="steps", flow="tube", nx=83, ny=2, Kn=0.002, N_ref=50,
             precision="mixed", order=1, sampling="energy_matched", K=0, steps=2),
        # the shock-tube configuration from its initial field: binary64, 20 steps
        dict(name="run_tube_9600_fp64_o1", kind="run", flow="tube", nx=100, ny=4, Kn=0.01, N_ref=50,
             precision="fp64", order=1, sampling="energy_matched", K=0, steps=20),
        # the benchmark's cavity in its settled state
        dict(name="steps_cavity_24_mixed_o2", kind="steps", flow="cavity", nx=24, ny=24, Kn=0.075, N_ref=100,
             precision="mixed", order=2, sampling="maxwell", K=0, steps=2),
        # the same flow in plain binary64 (odd size)
        dict(name="steps_cavity_21_fp64_o2", kind="steps", flow="cavity", nx=21, ny=21, Kn=0.075, N_ref=100,
             precision="fp64", order=2, sampling="maxwell", K=0, steps=2),
        # a large external-type flow (far-field ends, diffuse walls), first order
        dict(name="steps_channel_393k_mixed_o1", kind="steps", flow="channel", nx=64, ny=32, Kn=0.02, N_ref=60,
             precision="mixed", order=1, sampling="energy_matched", K=0, steps=2),
        # first-order g_p sampling
        dict(name="steps_cavity_16_mixed_gp1", kind="steps", flow="cavity", nx=16, ny=16, Kn=0.02, N_ref=100,
             precision="mixed", order=2, sampling="gp1", K=0, steps=2),
        # restart of a diatomic case (particles carry an internal energy): the
        # checkpoint from page-locked host arrays, one step, the fields read back
        dict(name="restart_cavity_15_mixed_K2", kind="restart", flow="cavity", nx=15, ny=15, Kn=0.075, N_ref=100,
             precision="mixed", order=2, sampling="maxwell", K=2),
        # independent instances of uneven size in one batch (tubes and cavities)
        dict(name="batch_14_mixed_o2", kind="batch", members=14, tets_lo=2000, tets_hi=30000, precision="mixed",
             order=2, sampling="energy_matched", steps=2),
        # gas-kinetic start-up with local time steps, second order
        dict(name="gks_channel_96k_o2_local", kind="gks", flow="channel", nx=40, ny=20, Kn=0.05, N_ref=60,
             precision="mixed", order=2, sampling="energy_matched", K=0, steps=4, local=True),
        # drag and heat-flux gradients, first and second order
        dict(name="adjoint_channel_40k_o1", kind="adjoint", flow="channel", nx=30, ny=15, Kn=0.05, N_ref=60,
             precision="mixed", order=1, sampling="energy_matched", K=0, steps=10, functional=0),
        dict(name="adjoint_channel_21k_o2", kind="adjoint", flow="channel", nx=24, ny=12, Kn=0.05, N_ref=60,
             precision="mixed", order=2, sampling="energy_matched", K=0, steps=4, functional=1),
        # reading the fields of a running case: W^p, W^h, primitives, Kn_GLL
        dict(name="fields_cavity_20_mixed", kind="fields", flow="cavity", nx=20, ny=20, Kn=0.075, N_ref=100,
             precision="mixed", order=2, sampling="maxwell", K=0),
    ]


def draw(rng):
    """One more case: a kind, then its sizes and options over their ranges."""
    kind = rng.choice(["steps"] * 6 + ["run", "batch", "gks", "adjoint", "fields", "restart"])

    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "batch":
        lo = rng.choice([2000, 3000, 5000])
        return dict(kind=kind, members=rng.randint(3, 17), tets_lo=lo, tets_hi=lo * rng.randint(3, 5),
                    precision=rng.choice(["mixed", "mixed", "fp64"]), order=rng.choice([1, 2]),
                    sampling="energy_matched", steps=rng.choice([2, 3, 4]))
    c = dict(kind=kind, precision=rng.choice(["mixed", "mixed", "fp64"]), order=rng.choice([1, 2]),
             sampling="energy_matched", K=0)
    c["flow"] = "channel" if kind == "adjoint" else rng.choice(["cavity", "channel", "tube"])
    if kind == "run":
        c["flow"] = "tube"
    lo, hi = (2000, 30000) if c["precision"] == "fp64" else (2000, 150000)
    if kind in ("adjoint", "run", "restart"):
        hi = min(hi, 30000)
    tets = logint(lo, hi)
    if c["flow"] == "cavity":
        c["nx"] = c["ny"] = max(6, int(round((tets / 6) ** (1 / 3))))
        c["Kn"] = round(math.exp(rng.uniform(math.log(0.005), math.log(0.075))), 4)
        c["N_ref"] = 100
        c["sampling"] = rng.choice(["maxwell", "energy_matched"])
        if c["order"] == 2 and rng.random() < 0.25:
            c["sampling"] = "gp1"
        elif c["sampling"] == "maxwell" and rng.random() < 0.4:
            c["K"] = rng.choice([1, 2, 5])
    elif c["flow"] == "channel":
        c["ny"] = max(4, int(round((tets / 12) ** (1 / 3))))
        c["nx"] = 2 * c["ny"] + rng.randint(-1, 1)
        c["Kn"] = round(math.exp(rng.uniform(math.log(0.005), math.log(0.05))), 4)
        c["N_ref"] = rng.choice([60, 100])
    else:
        c["ny"] = rng.randint(2, 5)
        c["nx"] = max(40, int(round(min(tets, 20000) / (6 * c["ny"] ** 2))))
        c["Kn"] = round(math.exp(rng.uniform(math.log(0.003), math.log(0.03))), 4)
        c["N_ref"] = 50
    if kind == "steps":
        c["steps"] = rng.choice([1, 2, 3, 4])
    elif kind == "run":
        c["steps"] = rng.randint(10, 20)
    elif kind == "gks":
        c.update(steps=rng.randint(2, 6), local=rng.random() < 0.5)
    elif kind == "adjoint":
        c.update(steps=rng.randint(2, 8) if c["order"] == 1 else rng.randint(1, 4), functional=rng.choice([0, 1]))
    return c


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=8)
def _flow(flow, nx, ny, Kn, N_ref, precision, order, K):
    if flow == "tube":
        return wl.shock_tube(nx=nx, ny=ny, nz=ny, Kn=Kn, N_ref=N_ref, precision=precision, order=order, K=K,
                             width=ny / nx)
    if flow == "cavity":
        return wl.cavity(n=nx, Kn=Kn, N_ref=N_ref, precision=precision, order=order, K=K)
    return wl.wall_channel(n=(nx, ny, ny), Kn=Kn, N_ref=N_ref, precision=precision, order=order)


@functools.lru_cache(maxsize=4)
def _instances(n, lo, hi, precision, order, sampling):
    """The benchmark's batch instances; their Knudsen numbers and velocities
    kept to where a population of a few N_ref per cell is the settled one."""
    out = wl.batch_instances(n=n, tets_lo=lo, tets_hi=hi, precision=precision, order=order, sampling=sampling)
    rng = np.random.default_rng(11)
    cfgs = []
    for k, c in enumerate(out):
        Kn = float(np.exp(rng.uniform(np.log(1e-3), np.log(0.03 if k % 2 == 0 else 0.075))))
        nc = len(c["mesh"]["tets"])
        if k % 2 == 0:
            ny = max(2, int(round((nc / 150.0) ** (1 / 3))))
            nx = max(4, int(round(nc / (6.0 * ny * ny))))
            c = wl.shock_tube(nx=nx, ny=ny, nz=ny, Kn=Kn, N_ref=50, precision=precision, order=order, width=ny / nx)
        else:
            m = max(3, int(round((nc / 6.0) ** (1 / 3))))
            c = wl.cavity(n=m, Kn=Kn, N_ref=100, precision=precision, order=order)
        c["params"]["sampling"] = sampling
        cfgs.append(c)
    return cfgs


def _config(case):
    c = _flow(case["flow"], case["nx"], case["ny"], case["Kn"], case["N_ref"], case["precision"], case["order"],
              case["K"])
    p = dict(c["params"], sampling=case["sampling"], K=case["K"])
    return {"mesh": c["mesh"], "W0": c["W0"], "params": p}


def _geometry(mesh):
    """Volumes [nc], projected areas [3, nc] and the largest edge extent."""
    x = mesh["nodes"][mesh["tets"]]
    a, b, c = x[:, 1] - x[:, 0], x[:, 2] - x[:, 0], x[:, 3] - x[:, 0]
    vol = np.abs(np.einsum("ij,ij->i", a, np.cross(b, c))) / 6.0
    s = np.zeros((3, len(vol)))
    for f in ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2)):
        s += 0.25 * np.abs(np.cross(x[:, f[1]] - x[:, f[0]], x[:, f[2]] - x[:, f[0]])).T
    return vol, s, float((x.max(axis=1) - x.min(axis=1)).max())


def _population(cfg):
    """Per cell: particles left after a settled step (even), the samples of a
    step and the fraction of the gas that collides in a step."""
    p, W = cfg["params"], cfg["W0"]
    vol, dS, _ = _geometry(cfg["mesh"])
    U = np.abs(W[1:4] / W[0])
    pr = (W[4] - 0.5 * (W[1:4] ** 2).sum(0) / W[0]) / (1.5 + 0.5 * p.get("K", 0))
    T = pr / W[0]
    dt = p["CFL"] * (vol / ((U + 3.0 * np.sqrt(T)) * dS).sum(0)).min()
    h = -np.expm1(-dt * pr / (p["mu_ref"] * T ** p["omega"]))
    sam = 2.0 * np.ceil(h / (1.0 + h) * p["N_ref"] / 2.0)
    left = 2 * np.rint(0.5 * sam * (1.0 - h) / h).astype(np.int64)
    return left, sam, h


def _with_capacity(cfg):
    """Room for the settled population where every cell samples a pair more:
    a step's survivor buckets (sized before collisions) and its samples."""
    _, sam, h = _population(cfg)
    cfg["params"]["particle_capacity"] = int(1.35 * ((sam + 2.0) * (1.0 + 1.0 / h)).sum() + 12 * len(h) + 8192)
    return cfg


def _perturbed(W0, mesh, K, seed):
    """The initial field with a smooth disturbance of 2 per cent (density and
    pressure), from the seed."""
    rng = np.random.default_rng(seed)
    c = mesh["nodes"][mesh["tets"]].mean(axis=1)
    s = np.zeros((2, len(c)))
    for _ in range(4):
        k, ph = rng.integers(1, 4, size=3), rng.uniform(0.0, 2.0 * np.pi, size=2)
        s += 0.005 * np.sin(2.0 * np.pi * (c @ k)[None] + ph[:, None])
    rho, U = W0[0] * (1.0 + s[0]), W0[1:4] / W0[0]
    e = 1.5 + 0.5 * K
    p = (W0[4] - 0.5 * W0[0] * (U * U).sum(0)) / e * (1.0 + s[1])
    return np.concatenate([rho[None], rho * U, (0.5 * rho * (U * U).sum(0) + e * p)[None]])


def _image(cfg, exps, seed):
    """The state image of a settled case (binary64, as import_state takes it),
    and the same on the device."""
    p, mesh = cfg["params"], cfg["mesh"]
    K, mixed = p.get("K", 0), p["precision"] == "mixed"
    g = torch.Generator(device="cuda").manual_seed(seed)
    dev = dict(device="cuda", dtype=torch.float64)
    vol, _, ext = _geometry(mesh)
    left, _, h = _population(cfg)
    vol, h, left = torch.tensor(vol, **dev), torch.tensor(h, **dev), torch.tensor(left, device="cuda")
    # each cell's number varies around the settled one
    n = 2 * torch.clamp((0.5 * left * (0.9 + 0.2 * torch.rand(len(vol), generator=g, **dev))).round(), max=16000).long()
    W = torch.tensor(cfg["W0"], **dev)
    nc, N = len(vol), int(n.sum())
    rho, U = W[0], W[1:4] / W[0]
    T = (W[4] - 0.5 * rho * (U * U).sum(0)) / ((1.5 + 0.5 * K) * rho)
    cell = torch.repeat_interleave(torch.arange(nc, device="cuda"), n)
    k = torch.arange(N, device="cuda") - (torch.cumsum(n, 0) - n)[cell]
    real = torch.float32 if mixed else torch.float64
    # velocities in pairs U +- sqrt(RT) X
    X = torch.randn(3, (N + 1) // 2, generator=g, **dev).repeat_interleave(2, dim=1)[:, :N]
    sig = torch.sqrt(T)
    u = (U[:, cell] + torch.where(k % 2 == 0, 1.0, -1.0) * sig[cell] * X).to(real).double()
    # positions uniform in the tet, on a grid that both precisions hold exactly
    w = torch.empty(4, N, **dev).exponential_(generator=g)
    w /= w.sum(0)
    nodes, tets = torch.tensor(mesh["nodes"], **dev), torch.tensor(mesh["tets"], device="cuda").long()
    x = torch.zeros(3, N, **dev)
    for j in range(4):
        x += w[j] * nodes[tets[:, j]].t()[:, cell]
    q = 2.0 ** (22 - math.ceil(math.log2(ext)))
    x = torch.round(x * q) / q
    m = ((1.0 - h) * rho * vol / n.clamp(min=1))[cell]
    e = torch.zeros(N, **dev)
    for _ in range(K):
        e += T[cell] * torch.randn(N, generator=g, **dev) ** 2
    e = e.to(real).double()
    phi = torch.stack([m, m * u[0], m * u[1], m * u[2], 0.5 * m * ((u * u).sum(0) + e)], dim=1)
    Wp = torch.segment_reduce(phi, "sum", lengths=n, axis=0).t() / vol
    held = n > 0
    hw = torch.where(held, h, torch.ones_like(h))
    Wn = Wp + torch.cat([(hw * rho)[None], hw * W[1:4], (hw * W[4])[None]])
    born = STEP - 1 - torch.randint(0, 200, (N,), generator=g, device="cuda")
    ident = (born << 40) | (cell << 16) | k
    dimg = dict(W=Wn, Wp=Wp, cell=cell, m=m, u=u, e=e, n=n)
    img = dict(W=Wn.cpu().numpy(), id=ident.cpu().numpy().astype(np.uint64), cell=cell.int().cpu().numpy(),
               x=x.cpu().numpy(), u=u.cpu().numpy(), m=m.cpu().numpy(), e=e.cpu().numpy(), step=STEP, t=0.0,
               exps=np.array(exps, dtype=np.int64))
    return img, dimg


def _simulation(cfg, seed):
    p = dict(cfg["params"], seed=1 + seed % (1 << 40))
    s = ugkwp.Simulation(cfg["mesh"], cfg["W0"], p, stream=torch.cuda.Stream())
    s.exps = list(ugkwp.ugkwp_state_info(s.handle).exps)
    return s


def _pinned(img):
    out = dict(img)
    for k, a in img.items():
        if isinstance(a, np.ndarray) and a.size > 16:
            t = torch.empty(a.nbytes, dtype=torch.uint8, pin_memory=True)
            b = t.numpy().view(a.dtype).reshape(a.shape)
            b[...] = a
            out[k] = b
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sims, outs = [], []
        for k, c in enumerate(_instances(case["members"], case["tets_lo"], case["tets_hi"], case["precision"],
                                         case["order"], case["sampling"])):
            c = _with_capacity({"mesh": c["mesh"], "W0": c["W0"], "params": dict(c["params"])})
            s = _simulation(c, seed + 1000 * k)
            s.set_state(_image(c, s.exps, seed + 1000 * k)[0])
            sims.append(s)
            outs.append(torch.empty(5, s.n_cells, dtype=torch.float64, device="cuda"))
        torch.cuda.synchronize()
        return dict(case=case, sims=sims, batch=ugkwp.Batch(sims), outs=outs)
    cfg = _with_capacity(_config(case))
    if kind in ("run", "gks"):
        cfg["W0"] = _perturbed(cfg["W0"], cfg["mesh"], case["K"], seed)
    s = _simulation(cfg, seed)
    st = dict(case=case, sim=s, tags=[1])
    if kind == "run":
        z = np.zeros(0)
        st["start"] = dict(W=cfg["W0"], id=z.astype(np.uint64), cell=z.astype(np.int32), x=np.zeros((3, 0)),
                           u=np.zeros((3, 0)), m=z, e=z, step=0, t=0.0, exps=np.array(s.exps))
    elif kind != "gks":
        img = _image(cfg, s.exps, seed)[0]
        s.set_state(img)
        if kind == "restart":
            st["image"] = _pinned(s.state_native())
    if kind == "fields":
        st["out"] = [torch.empty(5, s.n_cells, dtype=torch.float64, device="cuda") for _ in range(3)]
    else:
        st["out"] = torch.empty(5, s.n_cells, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return st


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "batch":
        st["batch"].step(c["steps"])
        st["batch"].sync()
        return [s.moments(ugkwp.W, out=o) for s, o in zip(st["sims"], st["outs"])]
    s = st["sim"]
    if kind == "steps":
        s.step(c["steps"])
        return s.moments(ugkwp.W, out=st["out"])
    if kind == "run":
        s.set_state(st["start"])
        n = s.step(c["steps"], stats=True)
        return [s.moments(ugkwp.W, out=st["out"]), n["n_particles"], n["n_sampled"], n["n_collided"], n["n_movers"],
                n["t"]]
    if kind == "gks":
        s.gks_steps(c["steps"], local_dt=c["local"])
        return s.moments(ugkwp.W, out=st["out"])
    if kind == "adjoint":
        a = s.adjoint(c["functional"], c["steps"], st["tags"])
        return [a, s.moments(ugkwp.W, out=st["out"])]
    if kind == "restart":
        s.set_state_native(st["image"])
        s.step(1)
        return s.moments(ugkwp.W)
    wp, wh, prim = st["out"]
    s.moments(ugkwp.WP, out=wp)
    s.moments(ugkwp.WH, out=wh)
    s.moments(ugkwp.PRIM, out=prim)
    return [wp, wh, prim, ugkwp.ugkwp_kn_gll(s.handle, s.n_cells)]


# -------------------------------------------------- work and exact values
def _step_work(cfg, steps, fresh=False):
    """Every particle's record read once and every survivor's written once, a
    cell's state read and written and its tet's record read once; the wave
    flux's binary64 arithmetic and about 100 operations per particle move."""
    p = cfg["params"]
    left, sam, _ = _population(cfg)
    if fresh:  # from the initial field: about N_ref particles per cell
        left = np.minimum(left, p["N_ref"])
    rec = (44 if p["precision"] == "mixed" else 68) + (0 if not p.get("K") else 4 if p["precision"] == "mixed" else 8)
    trk = 128 if p["precision"] == "mixed" else 144
    nc = len(left)
    nf = 2 * nc + len(cfg["mesh"]["bfaces"]) // 2
    moves = float((left + sam).sum())
    b = rec * (2.0 * float(left.sum())) + nc * (80.0 + trk) + nf * 36.0
    f = nf * (2500.0 if p["order"] == 2 else 400.0) + 100.0 * moves
    return {"bytes": steps * b, "flops": steps * f}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_step_work(c, case["steps"]) for c in _instances(case["members"], case["tets_lo"], case["tets_hi"],
                                                               case["precision"], case["order"], case["sampling"])]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    cfg = _config(case)
    nc = len(cfg["mesh"]["tets"])
    nf = 2 * nc + len(cfg["mesh"]["bfaces"]) // 2
    o2 = case["order"] == 2
    if kind in ("steps", "run"):
        return _step_work(cfg, case["steps"], kind == "run")
    if kind == "gks":
        # a cell's W read and written, its reconstruction weights and each face's geometry read
        return {"bytes": case["steps"] * (nc * (80.0 + (200.0 if o2 else 0.0)) + nf * 44.0),
                "flops": case["steps"] * nf * (2500.0 if o2 else 400.0)}
    if kind == "adjoint":
        # the recorded steps, the frozen forward and a reverse sweep of four times its arithmetic
        w = _step_work(cfg, case["steps"])
        f = nf * (2500.0 if o2 else 400.0)
        return {"bytes": w["bytes"] + case["steps"] * (nc * 400.0 + nf * 88.0), "flops": w["flops"] + case["steps"] * 5 * f}
    left = float(_population(cfg)[0].sum())
    if kind == "restart":
        w = _step_work(cfg, 1)
        return {"bytes": w["bytes"] + 44.0 * left, "flops": w["flops"]}
    r = 4 if case["precision"] == "mixed" else 8
    return {"bytes": left * (12.0 + 3 * r + (r if case["K"] else 0)) + nc * 8.0 * (5 * 4 + 1 + 12), "flops": 20.0 * left}


def exact(case, seed):
    """The particle steps draw from the library's own random streams, so their
    outputs have no value that plain arithmetic gives; the start-up steps and
    the fields have."""
    if case["kind"] == "gks":
        cfg = _with_capacity(_config(case))
        return _Gks(cfg, _perturbed(cfg["W0"], cfg["mesh"], case["K"], seed), case["local"]).run(case["steps"])
    if case["kind"] == "fields":
        cfg = _with_capacity(_config(case))
        d = _image(cfg, [0] * 5, seed)[1]
        W, K = d["W"], case["K"]
        U = W[1:4] / W[0]
        T = (W[4] - 0.5 * W[0] * (U * U).sum(0)) / ((1.5 + 0.5 * K) * W[0])
        G = _Gks(cfg, W.cpu().numpy(), False)
        g = torch.einsum("ikd,ik->id", G.lsq, G.values(W)[0] - W[0][:, None])
        p, om = cfg["params"], cfg["params"]["omega"]
        l = (2 * (5 - 2 * om) * (7 - 2 * om) / 15) * p["mu_ref"] * T ** om / (W[0] * torch.sqrt(2 * math.pi * T))
        return [d["Wp"], W - d["Wp"], torch.cat([W[:1], U, T[None]]), l * g.norm(dim=1) / W[0]]
    return None


PSI = [{(0, 0, 0): 1.0}, {(1, 0, 0): 1.0}, {(0, 1, 0): 1.0}, {(0, 0, 1): 1.0},
       {(2, 0, 0): 0.5, (0, 2, 0): 0.5, (0, 0, 2): 0.5}]


def _times(a, b):
    out = {}
    for p, v in a.items():
        for q, w in b.items():
            k = (p[0] + q[0], p[1] + q[1], p[2] + q[2])
            out[k] = out.get(k, 0.0) + v * w
    return out


class _Gks:
    """Steps of the gas-kinetic scheme without particles (monatomic or K
    internal degrees of freedom at first order of the wall's closed forms):
    least-squares gradients with Venkatakrishnan's limiter, moments of
    Maxwellians summed monomial by monomial, micro slopes by elimination."""

    def __init__(self, cfg, W0, local):
        self.p, self.local = cfg["params"], local
        t = dict(device="cuda", dtype=torch.float64)
        mesh = cfg["mesh"]
        self.W = torch.tensor(W0, **t)
        vol, dS, _ = _geometry(mesh)
        self.vol, self.dS = torch.tensor(vol, **t), torch.tensor(dS, **t)
        nodes, tets = np.asarray(mesh["nodes"]), np.asarray(mesh["tets"], dtype=np.int64)
        nc, nn = len(tets), len(nodes)

        def key(f):
            f = np.sort(f.astype(np.int64), axis=1)
            return (f[:, 0] * nn + f[:, 1]) * nn + f[:, 2]

        fl = tets[:, [[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]]]  # [nc, 4, 3]
        ks = key(fl.reshape(-1, 3))
        order = np.argsort(ks, kind="stable")
        twin = np.full(4 * nc, -1, dtype=np.int64)
        same = ks[order[1:]] == ks[order[:-1]]
        twin[order[1:][same]], twin[order[:-1][same]] = order[:-1][same], order[1:][same]
        kb = key(np.asarray(mesh["bfaces"]))
        ob = np.argsort(kb)
        at = np.minimum(np.searchsorted(kb[ob], ks), len(kb) - 1)
        self.tag = torch.tensor(np.where(twin < 0, np.asarray(mesh["btags"])[ob][at], -1).reshape(nc, 4), device="cuda")
        twin = torch.tensor(twin.reshape(nc, 4), device="cuda")
        self.nb = torch.where(twin >= 0, twin // 4, -1)
        x = torch.tensor(nodes[tets], **t)
        xf = torch.tensor(nodes[fl], **t)  # [nc, 4, 3, 3]
        c = x.mean(1)
        a = 0.5 * torch.linalg.cross(xf[:, :, 1] - xf[:, :, 0], xf[:, :, 2] - xf[:, :, 0])
        fc = xf.mean(2)
        a = torch.where(((fc - c[:, None]) * a).sum(-1, keepdim=True) < 0, -a, a)
        self.area = a.norm(dim=-1)
        self.n = a / self.area[..., None]  # outward
        self.dxf = fc - c[:, None]
        h = (self.dxf * self.n).sum(-1, keepdim=True)
        dx = torch.where((self.nb >= 0)[..., None], c[self.nb.clamp(min=0)] - c[:, None], 2.0 * h * self.n)
        w = 1.0 / (dx * dx).sum(-1)
        A = torch.einsum("ik,ikd,ike->ide", w, dx, dx)
        self.lsq = torch.einsum("ide,ike,ik->ikd", torch.linalg.inv(A), dx, w)
        self.eps2 = (self.p["venkat_K"] * self.vol ** (1.0 / 3.0)) ** 3
        self.own = torch.nonzero(((self.nb >= 0) & (self.nb > torch.arange(nc, device="cuda")[:, None])).reshape(-1))[:, 0]
        self.twin = twin.reshape(-1)[self.own]
        self.e = 1.5 + 0.5 * self.p.get("K", 0)
        self.K = float(self.p.get("K", 0))

    def values(self, W):
        """The neighbours' values [q, nc, 4], with the ghosts of the boundary faces."""
        v = W[:, self.nb.clamp(min=0)]
        own = W[:, :, None].expand_as(v)
        g = own.clone()
        for k, b in enumerate(self.p["bc"]):
            at = self.tag == k
            if b["type"] == "specular":
                mn = (own[1:4] * self.n.permute(2, 0, 1)).sum(0)
                g[1:4] = torch.where(at, own[1:4] - 2.0 * mn * self.n.permute(2, 0, 1), g[1:4])
            elif b["type"] == "farfield":
                g = torch.where(at, torch.tensor(b["W_in"], device="cuda", dtype=torch.float64)[:, None, None], g)
        return torch.where(self.nb >= 0, v, g)

    def prim(self, W):
        U = W[1:4] / W[0]
        pr = (W[4] - 0.5 * W[0] * (U * U).sum(0)) / self.e
        return U, pr, pr / W[0]

    def tau(self, T, pr):
        return self.p["mu_ref"] * T ** self.p["omega"] / pr

    def gradients(self, W):
        v = self.values(W)
        d = v - W[:, :, None]
        g = torch.einsum("ikd,qik->qid", self.lsq, d)
        d2 = torch.einsum("qid,ikd->qik", g, self.dxf)
        hi, lo = d.amax(-1).clamp(min=0.0), d.amin(-1).clamp(max=0.0)
        d1 = torch.where(d2 > 0, hi[..., None], lo[..., None])
        e = self.eps2[None, :, None]
        r = ((d1 * d1 + e) * d2 + 2.0 * d2 * d2 * d1) / (d2 * (d1 * d1 + 2.0 * d2 * d2 + d1 * d2 + e))
        r = torch.where(d2 == 0.0, torch.ones_like(r), r)
        return g * r.amin(-1).clamp(max=1.0)[..., None]

    class Gauss:
        """Moments of the unit Maxwellian (U in the face frame, theta = RT)."""

        def __init__(s, U, th, half):
            def table(mean, m0, m1):
                M = [m0, m1]
                for k in range(7):
                    M.append(mean * M[k + 1] + (k + 1) * th * M[k])
                return M

            one = torch.ones_like(th)
            if half:
                z = U[0] / torch.sqrt(2.0 * th)
                m0 = 0.5 * torch.special.erfc(-half * z)
                m1 = U[0] * m0 + half * torch.exp(-z * z) * torch.sqrt(th / (2.0 * math.pi))
            else:
                m0, m1 = one, U[0]
            s.t = [table(U[0], m0, m1), table(U[1], one, U[1]), table(U[2], one, U[2])]

        def of(s, poly):
            return sum(v * s.t[0][k[0]] * s.t[1][k[1]] * s.t[2][k[2]] for k, v in poly.items())

        def psi(s, w):
            return torch.stack([s.of(_times(w, q)) for q in PSI])

        def slope(s, w, a):
            return torch.stack([sum(a[j] * s.of(_times(w, _times(PSI[j], q))) for j in range(5)) for q in PSI])

        def solve(s, b):
            M = torch.stack([torch.stack([s.of(_times(p, q)) for q in PSI], -1) for p in PSI], -2)
            return torch.linalg.solve(M, b.movedim(0, -1).unsqueeze(-1)).squeeze(-1).movedim(-1, 0)

    def frame(self, n):
        a = torch.zeros_like(n)
        a[torch.arange(len(n), device="cuda"), n.abs().argmin(1)] = 1.0
        t1 = torch.linalg.cross(a, n)
        t1 = t1 / t1.norm(dim=1, keepdim=True)
        return torch.stack([n, t1, torch.linalg.cross(n, t1)], dim=1)  # [f, row, xyz]

    @staticmethod
    def rotate(R, W):
        return torch.cat([W[:1], torch.einsum("frx,xf->rf", R, W[1:4]), W[4:5]])

    def coefficients(self, dt, tau):
        e = torch.exp(-dt / tau)
        q4 = -tau * torch.expm1(-dt / tau)
        return (dt - q4, 2.0 * tau * q4 - tau * dt * (1.0 + e), 0.5 * dt * dt - tau * dt + tau * q4, q4,
                tau * dt * e - tau * q4)

    def flux(self, WL, WR, gL, gR, n, dt):
        """Flux along n (per unit area) from two states and their slopes [q, f, xyz]."""
        R = self.frame(n)
        ux = {(1, 0, 0): 1.0}
        dirs = [{(2, 0, 0): 1.0}, {(1, 1, 0): 1.0}, {(1, 0, 1): 1.0}]
        W0, G, S, B = 0.0, 0.0, 0.0, 0.0
        for W, g, half in ((WL, gL, 1), (WR, gR, -1)):
            Wr = self.rotate(R, W)
            U, _, T = self.prim(Wr)
            M = self.Gauss(U, T, half)
            W0 = W0 + Wr[0] * M.psi({(0, 0, 0): 1.0})
            G = G + Wr[0] * M.psi(ux)
            if g is not None:
                F = self.Gauss(U, T, 0)
                s = torch.stack([self.rotate(R, torch.einsum("qfx,fx->qf", g, R[:, d])) for d in range(3)])
                B = B + 0.5 * s
                for d in range(3):
                    S = S + Wr[0] * M.slope(dirs[d], F.solve(s[d] / Wr[0]))
        U, pr, T = self.prim(W0)
        q1, q2, q3, q4, q5 = self.coefficients(dt, self.tau(T, pr))
        M = self.Gauss(U, T, 0)
        F = q1 * W0[0] * M.psi(ux) + q4 * G
        if gL is not None:
            a = [M.solve(B[d] / W0[0]) for d in range(3)]
            one = [{(1, 0, 0): 1.0}, {(0, 1, 0): 1.0}, {(0, 0, 1): 1.0}]
            A = M.solve(-sum(M.slope(one[d], a[d]) for d in range(3)))
            F = F + q5 * S + W0[0] * (q2 * sum(M.slope(dirs[d], a[d]) for d in range(3)) + q3 * M.slope(ux, A))
        return torch.cat([F[:1], torch.einsum("frx,rf->xf", R, F[1:4]), F[4:5]])

    def run(self, steps):
        if self.K:
            return None  # the internal moments are not written out here
        W, nc = self.W, self.W.shape[1]
        for _ in range(steps):
            U, pr, T = self.prim(W)
            dtc = self.p["CFL"] * self.vol / ((U.abs() + 3.0 * torch.sqrt(T)) * self.dS).sum(0)
            if not self.local:
                dtc = dtc.min().expand(nc)
            o2 = self.p["order"] == 2
            g = self.gradients(W) if o2 else None
            acc = torch.zeros(5, 4 * nc, device="cuda", dtype=torch.float64)
            # interior faces, each once
            i, j = self.own // 4, self.twin // 4
            n = self.n.reshape(-1, 3)[self.own]
            dt = torch.minimum(dtc[i], dtc[j])
            WL, WR, gL, gR = W[:, i], W[:, j], None, None
            if o2:
                gL, gR = g[:, i], g[:, j]
                WL = WL + torch.einsum("qfx,fx->qf", gL, self.dxf.reshape(-1, 3)[self.own])
                WR = WR + torch.einsum("qfx,fx->qf", gR, self.dxf.reshape(-1, 3)[self.twin])
            F = self.flux(WL, WR, gL, gR, n, dt) / dt
            acc[:, self.own], acc[:, self.twin] = F, -F
            # boundary faces at first order
            for k, b in enumerate(self.p["bc"]):
                at = torch.nonzero((self.tag == k).reshape(-1))[:, 0]
                if not len(at):
                    continue
                i, n = at // 4, self.n.reshape(-1, 3)[at]
                dt, Wi = dtc[i], W[:, i]
                if b["type"] == "farfield":
                    Wr = torch.tensor(b["W_in"], device="cuda", dtype=torch.float64)[:, None].expand_as(Wi)
                    F = self.flux(Wi, Wr, None, None, n, dt)
                elif b["type"] == "specular":
                    mn = (Wi[1:4] * n.t()).sum(0)
                    Wr = torch.cat([Wi[:1], Wi[1:4] - 2.0 * mn * n.t(), Wi[4:5]])
                    F = self.flux(Wi, Wr, None, None, n, dt)
                    fn = (F[1:4] * n.t()).sum(0)
                    F = torch.cat([torch.zeros_like(F[:1]), fn * n.t(), torch.zeros_like(F[:1])])
                else:
                    R = self.frame(n)
                    Wr = self.rotate(R, Wi)
                    Uf, pf, Tf = self.prim(Wr)
                    q1, _, _, q4, _ = self.coefficients(dt, self.tau(Tf, pf))
                    Gin = (q1 + q4) * Wr[0] * self.Gauss(Uf, Tf, 1).psi({(1, 0, 0): 1.0})
                    Uw = torch.einsum("frx,x->rf", R, torch.tensor(b["U_w"], device="cuda", dtype=torch.float64))
                    Gw = self.Gauss(Uw, torch.full_like(Tf, b["T_w"]), -1).psi({(1, 0, 0): 1.0})
                    F = Gin - Gin[0] / Gw[0] * Gw
                    F = torch.cat([F[:1], torch.einsum("frx,rf->xf", R, F[1:4]), F[4:5]])
                acc[:, at] = F / dt
            W = W - dtc * (acc * self.area.reshape(-1)).reshape(5, nc, 4).sum(-1) / self.vol
        return W
