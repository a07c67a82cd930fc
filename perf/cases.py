"""The work that programs have this library do, as cases to be measured.

Each case stands for one real use (the comments in `listed` say which): a pass
is what such a program repeats - some coupled time steps through `lbm_step`
followed by the reads it samples, or one call of the force surrogate.

`exact` restates the method (arXiv 2505.10171: pull streaming with bounce-back,
colour-gradient order parameter, geometric wetting, MRT collision with Guo
forcing, momentum exchange, capillary force, DEM, refill) and the surrogate
network in plain 64-bit torch, whole arrays at a time.
"""
import math
import random

import numpy as np
import torch

from paper_2505_10171_gb300 import lbm
from paper_2505_10171_gb300 import workloads as W

KEEP = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float32, "bf16": torch.float32}
# the velocity is formed from the population offsets alone: it is kept in their type
KEEP_U = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
F64 = torch.float64


def listed():
    return [
        # the parity configuration (48x32x32, drop R=10, one sphere R=4, sliding wall), stepped one step at a time with
        # the forces read after each: the smallest calls, where launches and latency count
        dict(name="parity_step_fp64", kind="coupled", precision="fp64", nx=48, ny=32, nz=32, spheres=1, radius=4.0,
             steps=1, slide=1),
        # a coarse drop-sphere run watched step by step (every step's forces and the order parameter)
        dict(name="watched_step_fp32", kind="coupled", precision="fp32", nx=128, ny=64, nz=64, spheres=8, radius=4.0,
             steps=1),
        # a single collision of the friction study on a ragged lattice, bfloat16 storage
        dict(name="ragged_bf16", kind="coupled", precision="bf16", nx=201, ny=91, nz=37, spheres=3, radius=5.0, steps=16),
        # the resolved run (256x128x128, drop R=40, eight spheres R=8), sampled every 16 steps
        dict(name="resolved_fp32", kind="coupled", precision="fp32", nx=256, ny=128, nz=128, spheres=8, radius=8.0,
             steps=16),
        # the same with 16-bit offset storage
        dict(name="resolved_fp16", kind="coupled", precision="fp16", nx=256, ny=128, nz=128, spheres=8, radius=8.0,
             steps=16),
        # particle migration in the periodic body-force tube (64x64x1024), velocity sampled
        dict(name="tube_fp32", kind="tube", precision="fp32", tube=31, nz=1024, radius=6.0, steps=16, faces=0),
        # the pressure-driven tube of the migration benchmark (radius 40), a shorter piece
        dict(name="pressure_tube_fp32", kind="tube", precision="fp32", tube=40, nz=640, radius=12.2, steps=16, faces=1),
        # the friction map: 36 collisions of 200x90x36 in one context, shells sampled
        dict(name="friction_map_fp16", kind="map", precision="fp16", count=36, scale=0.5, steps=16),
        # the parameter sweep: 96 uneven domains in one context
        dict(name="sweep_fp16", kind="sweep", precision="fp16", count=96, rmin=16.0, rmax=40.0, steps=4),
        # 64 coarse runs (96x48x48, eight held spheres each) with the force surrogate in the step
        dict(name="coarse_surrogate_fp32", kind="coarse", precision="fp32", count=64, steps=16),
        # one epoch of the surrogate's training on a part of the campaign's samples
        dict(name="surrogate_train", kind="train", n=20000, batch=512),
        # the network evaluated on the 512 spheres of 64 runs
        dict(name="surrogate_predict", kind="predict", n=512),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["coupled", "coupled", "coupled", "tube", "map", "sweep", "coarse", "train", "predict", "gradient"])
    if kind == "coupled":
        precision = rng.choice(["fp64", "fp32", "fp16", "bf16"])
        nodes = _log(rng, 4e4, 5e5 if precision == "fp64" else 4.2e6)
        a = rng.uniform(1.4, 2.2)
        b = rng.uniform(0.7, 1.0)
        ny = max(32, round((nodes / (a * b)) ** (1.0 / 3.0)))
        nx, nz = max(48, round(a * ny)), max(28, round(b * ny))
        if rng.random() < 0.5:
            nx, ny, nz = nx // 2 * 2, ny // 2 * 2, nz // 2 * 2
        return dict(kind=kind, precision=precision, nx=nx, ny=ny, nz=nz, spheres=rng.choice([0, 1, 2, 4, 8]),
                    radius=round(min(rng.uniform(3.5, 8.0), ny / 10.0), 2), steps=rng.choice([1, 4, 16]),
                    slide=rng.choice([0, 0, 1]), buoyant=rng.choice([0, 0, 0, 1]))
    if kind == "tube":
        tube, faces = round(_log(rng, 15, 41)), rng.choice([0, 1])
        # between faces the sphere needs room for the steps that a run takes
        return dict(kind=kind, precision=rng.choice(["fp32", "fp32", "fp16"]), tube=tube,
                    nz=round(_log(rng, 256 if faces else 64, 1024)), radius=round(tube * rng.uniform(0.17, 0.31), 2),
                    steps=rng.choice([1, 8, 16]), faces=faces)
    if kind == "map":
        return dict(kind=kind, precision=rng.choice(["fp16", "fp32"]), count=round(_log(rng, 2, 36)),
                    scale=round(rng.uniform(0.45, 0.62), 3), steps=rng.choice([4, 16]))
    if kind == "sweep":
        rmin = rng.uniform(12.0, 18.0)
        return dict(kind=kind, precision=rng.choice(["fp16", "bf16", "fp32"]), count=round(_log(rng, 3, 48)),
                    rmin=round(rmin, 2), rmax=round(rng.uniform(rmin + 4.0, 40.0), 2), steps=rng.choice([1, 4]))
    if kind == "coarse":
        return dict(kind=kind, precision="fp32", count=round(_log(rng, 1, 64)), steps=rng.choice([1, 16]))
    if kind == "train":
        return dict(kind=kind, n=round(_log(rng, 300, 20000)), batch=rng.choice([64, 128, 300, 512, 1024]))
    return dict(kind=kind, n=round(_log(rng, 1, 4096 if kind == "gradient" else 20000)))


# ---------------------------------------------------------------------------
# set-ups: parameters, spheres and initial fields of every instance of a case
# ---------------------------------------------------------------------------
def _axes(p, device):
    z = torch.arange(p["nz"], dtype=F64, device=device)[:, None, None]
    y = torch.arange(p["ny"], dtype=F64, device=device)[None, :, None]
    x = torch.arange(p["nx"], dtype=F64, device=device)[None, None, :]
    return x, y, z


def _mi(d, n):
    """Minimum-image displacement on a periodic axis."""
    return d - n * torch.floor(d / n + 0.5)


def _drop_fields(p, centre, R, speed):
    """phi, rho, u of a drop with a tanh edge that moves at `speed` along x."""
    x, y, z = _axes(p, "cuda")
    r = torch.sqrt(_mi(x - centre[0], p["nx"]) ** 2 + _mi(y - centre[1], p["ny"]) ** 2 + _mi(z - centre[2], p["nz"]) ** 2)
    phi = torch.tanh(2.0 * (R - r) / W.INTERFACE_WIDTH)
    u = torch.zeros((3,) + phi.shape, dtype=F64, device="cuda")
    u[0] = speed * 0.5 * (1.0 + phi)
    if p["wall_z0"]:
        u[0, 0] = 0.0
    rho = 1.0 + 2.0 / 3.0 * 3.0 * p["sigma"] / R * 0.5 * (1.0 + phi)  # Laplace pressure inside
    return phi, rho, u


def _spheres(rng, p, n, R, x_lo):
    """At most n resting spheres ahead of the drop, clear of one another's contact:
    as many as fit, each at a random place of its own cell."""
    Rc = R + p["delta_R"]
    lo, hi = (x_lo, Rc + 1.0), (p["nx"] - Rc - 2.0, p["ny"] - Rc - 1.0)
    cell = 2.0 * Rc + 1.0
    cols, rows = (max(1, int((b - a) / cell) + 1) for a, b in zip(lo, hi))
    slack = [max(0.0, (b - a - (k - 1) * cell) / k) for a, b, k in zip(lo, hi, (cols, rows))]
    out = []
    for k in rng.sample(range(cols * rows), min(n, cols * rows)):
        c = [lo[d] + i * (cell + slack[d]) + rng.uniform(0.0, slack[d]) for d, i in ((0, k % cols), (1, k // cols))]
        out.append(dict(x=(c[0], c[1], R + 1.5), R=R, rho_p=W.PARTICLE_DENSITY, theta_deg=rng.uniform(30.0, 90.0)))
    return out


def _coupled(case, seed):
    rng = random.Random(seed)
    R_p = case["radius"]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    speed = rng.uniform(3e-3, 6e-3)
    p = dict(W.COMMON, nx=nx, ny=ny, nz=nz, wall_z0=1, theta_wall_deg=rng.uniform(90.0, 150.0), nu_a=1.0 / 6.0,
             nu_b=1.0 / 60.0, mu_s=0.3, mu_r=0.05, gn=W.resting_damping(R_p), body_force_a=(2.0e-6, 0.0, 0.0),
             g_particle=(0.0, 0.0, -10.0 * W.COMMON["sigma"] * R_p), drop_speed_control=1,
             drop_speed_target=(speed, 0.0, 0.0), drop_speed_interval=100)
    if case.get("slide"):
        p.update(wall_velocity=(1e-3, 0.0, 0.0), nu_b=1.0 / 6.0, drop_speed_control=0)
    if case.get("buoyant"):
        p.update(buoyancy_a=(0.0, 0.0, 1e-4))
    R_d = min(0.31 * ny, 0.6 * nz, 0.17 * nx) * rng.uniform(0.95, 1.0)
    xd = R_d + 4.0 + rng.uniform(0.0, 4.0)
    parts = _spheres(rng, p, case["spheres"], R_p, xd + R_d + R_p + 3.0)
    return [dict(p=p, parts=parts, fields=lambda: _drop_fields(p, (xd, ny / 2.0, 0.5), R_d, speed))]


def _tube(case, seed):
    rng = random.Random(seed)
    R_t, nz, nu, c = float(case["tube"]), case["nz"], 1.0 / 6.0, (2 * case["tube"] + 1) / 2.0
    n = 2 * case["tube"] + 2
    uc = rng.uniform(0.015, 0.025)
    # the set-ups' compressibility: the drop over the faces is that of the same flow
    g = 4.0 * nu * uc / R_t ** 2
    p = dict(W.COMMON, nx=n, ny=n, nz=nz, wall_z0=0, nu_a=nu, nu_b=nu, sigma=0.0, mu_s=0.0, mu_r=0.0, g_particle=(0.0, 0.0, 0.0))
    drho = 3.0 * g * (nz - 2 - 2 * W.FACE_SHIFT)
    if case["faces"]:
        p.update(pressure_z=1, rho_in=1.0 + drho / 2, rho_out=1.0 - drho / 2)
    else:
        p.update(body_force_a=(0.0, 0.0, g))
    l = rng.uniform(0.2, 0.35) * R_t
    parts = [dict(x=(c + l, c, nz * rng.uniform(0.4, 0.6)), R=case["radius"], rho_p=1.0, theta_deg=90.0,
                  v=(0.0, 0.0, uc * (1.0 - (l / R_t) ** 2)))]

    def fields():
        x, y, z = _axes(p, "cuda")
        r2 = (x - c) ** 2 + (y - c) ** 2 + 0.0 * z
        u = torch.zeros((3,) + r2.shape, dtype=F64, device="cuda")
        u[2] = torch.clamp(uc * (1.0 - r2 / R_t ** 2), min=0.0)
        rho = 1.0 + 0.0 * r2
        if case["faces"]:
            rho = rho + drho * (0.5 - (z - 1.0) / (nz - 3.0))
        return torch.ones_like(r2), rho, u

    y, x = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    mask = np.broadcast_to(((x - c) ** 2 + (y - c) ** 2 > R_t ** 2)[None], (nz, n, n))
    return [dict(p=dict(p, store_velocity=1), parts=parts, fields=fields, mask=mask)]


def _map(case, seed):
    rng, out = random.Random(seed), []
    s, sigma = case["scale"], 0.01
    for k in range(case["count"]):
        nx, ny, nz = int(round(400 * s)), int(round(181 * s)), int(round(71 * s))
        R_p, R_d = 10.0 * s, 50.0 * s
        g_p = 5.23 * sigma * R_p
        p = dict(W.COMMON, nx=nx, ny=ny, nz=nz, wall_z0=1, theta_wall_deg=90.0, sigma=sigma, nu_a=1.0 / 6.0,
                 nu_b=1.0 / 60.0, body_force_a=(1.25 * sigma / R_d ** 2, 0.0, 0.0), mu_s=rng.uniform(0.0, 1.0),
                 mu_r=rng.uniform(0.0, 1.0), gn=W.resting_damping(R_p), g_particle=(0.0, 0.0, -g_p), store_velocity=1)
        xd, speed = 1.0 + R_d + 6.0 * s, rng.uniform(2e-3, 5e-3)
        parts = [dict(x=(xd + R_d + R_p + 3.0 * rng.uniform(0.2, 1.0), ny / 2.0 + 0.5 * R_p,
                         0.5 + R_p + p["delta_R"] - g_p / p["kn"]), R=R_p, rho_p=W.PARTICLE_DENSITY, theta_deg=90.0)]
        out.append(dict(p=p, parts=parts, fields=lambda p=p, xd=xd, R_d=R_d, speed=speed: _drop_fields(
            p, (xd, p["ny"] / 2.0, 0.5), R_d, speed)))
    return out


def _sweep(case, seed):
    rng, out = random.Random(seed), []
    for k in range(case["count"]):
        R_d = random.Random(4242 + k).uniform(case["rmin"], case["rmax"])  # the same domains for every seed
        U = rng.uniform(1e-3, 1e-2)
        nx, ny, nz = max(96, W.ceil8(5.5 * R_d)), max(64, W.ceil8(3.2 * R_d)), max(64, W.ceil8(3.2 * R_d))
        R_p, sigma = R_d / 5.0, W.COMMON["sigma"]
        p = dict(W.COMMON, nx=nx, ny=ny, nz=nz, wall_z0=1, theta_wall_deg=90.0, nu_a=1.0 / 6.0, nu_b=1.0 / 60.0,
                 mu_s=rng.uniform(0.0, 0.6), mu_r=rng.uniform(0.0, 0.1), gn=W.resting_damping(R_p),
                 body_force_a=(U * 4e-4, 0.0, 0.0), g_particle=(0.0, 0.0, -10.0 * sigma * R_p), drop_speed_control=1,
                 drop_speed_target=(U, 0.0, 0.0), drop_speed_interval=100)
        xd = 1.2 * R_d
        parts = [dict(x=(xd + R_d + R_p + 3.0, ny / 2.0, R_p + 1.5), R=R_p, rho_p=W.PARTICLE_DENSITY, theta_deg=90.0)]
        out.append(dict(p=p, parts=parts, fields=lambda p=p, xd=xd, R_d=R_d, U=U: _drop_fields(
            p, (xd, p["ny"] / 2.0, 0.5), R_d, U)))
    return out


def _coarse(case, seed):
    rng, out, s = random.Random(seed), [], 3.0 / 8.0
    R_p, U, sigma = 3.0, 5.0e-3 * s, W.COMMON["sigma"] * s
    for k in range(case["count"]):
        p = dict(W.COMMON, nx=96, ny=48, nz=48, wall_z0=1, theta_wall_deg=150.0, nu_a=1.0 / 6.0, nu_b=1.0 / 60.0,
                 mu_s=0.3, mu_r=0.05, gn=W.resting_damping(R_p), sigma=sigma, body_force_a=(2.0e-6 * s, 0.0, 0.0),
                 g_particle=(0.0, 0.0, -2.0 * sigma * R_p), drop_speed_control=1, drop_speed_target=(U, 0.0, 0.0),
                 drop_speed_interval=100, store_velocity=1, surrogate_u_ref=U, surrogate_r_ref=R_p,
                 surrogate_shell_gap=0.5 * R_p)
        parts = []
        while len(parts) < 8:
            c = (rng.uniform(36.75, 57.0), rng.uniform(4.5, 43.5))
            if all((c[0] - q["x"][0]) ** 2 + (c[1] - q["x"][1]) ** 2 >= 72.0 for q in parts):
                parts.append(dict(x=(c[0], c[1], 4.5), R=R_p, rho_p=W.PARTICLE_DENSITY, theta_deg=rng.uniform(30.0, 90.0),
                                  kinematic=1))
        out.append(dict(p=p, parts=parts, fields=lambda p=p: _drop_fields(p, (18.0, 24.0, 0.5), 15.0, U)))
    return out


SETUPS = {"coupled": _coupled, "tube": _tube, "map": _map, "sweep": _sweep, "coarse": _coarse}


def _weights(seed):
    """Uniform weights of the network's fan-in, as the campaign starts from."""
    rng, th, o = np.random.default_rng(seed), np.zeros(lbm.MLP_PARAMS, dtype=np.float32), 0
    for rows, cols, fan in ((128, 400, 387), (128, 0, 0), (128, 128, 128), (128, 0, 0), (6, 128, 128), (6, 0, 0)):
        if cols:
            blk = rng.uniform(-1.0, 1.0, (rows, cols)) / math.sqrt(fan)
            if cols == 400:
                blk[:, 387:] = 0.0
            th[o:o + rows * cols] = blk.reshape(-1)
        o += rows * cols if cols else rows
    return th


def _samples(n, seed):
    """Shell features (phi and scaled velocities that vary along the shell) and force targets."""
    rng = np.random.default_rng(seed)
    X = np.empty((n, lbm.MLP_INPUTS), dtype=np.float32)
    shell = X[:, :384].reshape(n, 96, 4)
    t = np.linspace(-1.0, 1.0, 96, dtype=np.float32)[None, :]
    cut, width = rng.uniform(-2.0, 1.5, (n, 1)).astype(np.float32), rng.uniform(0.1, 0.6, (n, 1)).astype(np.float32)
    shell[:, :, 0] = np.tanh((cut - t) / width)
    shell[:, :, 1:] = rng.standard_normal((n, 1, 3), dtype=np.float32) * (1.0 + 0.3 * t)[:, :, None]
    shell[:, :, 1:] += 0.1 * rng.standard_normal((n, 96, 3), dtype=np.float32)
    th = rng.uniform(math.radians(30.0), math.radians(90.0), n)
    X[:, 384], X[:, 385], X[:, 386] = np.cos(th), np.sin(th), 1.0
    Y = np.stack([shell[:, :, k % 4].mean(1) + 0.3 * shell[:, (17 * k) % 96, 0] for k in range(6)], axis=1)
    return X, np.ascontiguousarray(Y, dtype=np.float32)


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
_STREAM = []


def _stream():
    """The program's one stream: its contexts and its own tensors work on it."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, s.stream = case, _stream()
    if case["kind"] in ("train", "predict", "gradient"):
        # the network lives in a context; a small coarse one hosts it
        s.ctx = lbm.Context(dict(W.COMMON, nx=16, ny=16, nz=16, store_velocity=1), "fp32", stream=s.stream.cuda_stream)
        s.ctx.lbm_surrogate_load(_weights(seed))
        s.X, s.Y = _samples(case["n"], seed)
        s.epoch = seed
        return s
    inst = SETUPS[case["kind"]](case, seed)
    with torch.cuda.stream(s.stream):
        s.ctx = lbm.Context([i["p"] for i in inst], case["precision"], stream=s.stream.cuda_stream)
        for k, i in enumerate(inst):
            if i.get("mask") is not None:
                s.ctx.lbm_set_solid_mask(i["mask"], inst=k)
            if i["parts"]:
                s.ctx.lbm_add_particles(i["parts"], inst=k)
            phi, rho, u = (t.contiguous() for t in i["fields"]())
            s.ctx.lbm_init_fields_device(phi.data_ptr(), rho.data_ptr(), u.data_ptr(), inst=k)
            s.stream.synchronize()
        if case["kind"] == "coarse":
            s.ctx.lbm_surrogate_load(_weights(seed))
            s.ctx.lbm_set_force_model(lbm.FORCE_SURROGATE)
        s.mask = lbm.FIELD_PHI if case["kind"] in ("sweep", "map", "coarse") else (
            lbm.FIELD_RHO_A | lbm.FIELD_RHO_B | lbm.FIELD_PHI)
        if case["kind"] == "tube":
            s.mask = lbm.FIELD_RHO_A | lbm.FIELD_U
        count = 1 if s.mask == lbm.FIELD_PHI else 3
        s.nodes = [s.ctx.num_nodes(k) for k in range(len(inst))]
        s.out = torch.zeros((4 if case["kind"] == "tube" else count) * sum(s.nodes), dtype=F64, device="cuda")
        s.ring = None
        total = sum(len(i["parts"]) for i in inst)
        if total:
            s.ring = torch.zeros((case["steps"], total, lbm.PARTICLE_RECORD), dtype=F64, device="cuda")
            s.stream.synchronize()
            s.ctx.lbm_set_record_ring((s.ring.data_ptr(), case["steps"]))
    return s


def run(s):
    case = s.case
    if case["kind"] == "predict":
        return s.ctx.lbm_surrogate_predict(s.X)
    if case["kind"] == "gradient":
        g, loss = s.ctx.lbm_surrogate_gradient(s.X, s.Y)
        return g, np.float32(loss)
    if case["kind"] == "train":
        loss = s.ctx.lbm_surrogate_train(s.X, s.Y, 1, case["batch"], 1e-3, s.epoch)
        s.epoch += 1
        return s.ctx.lbm_surrogate_save(), np.float32(loss)
    s.ctx.lbm_step(case["steps"])
    per = s.out.numel() // sum(s.nodes)
    with torch.cuda.stream(s.stream):
        at = 0
        for k, n in enumerate(s.nodes):
            s.ctx.lbm_read_fields_device(s.mask, s.out.data_ptr() + 8 * at, inst=k)
            at += per * n
        keep = KEEP[case["precision"]]
        got = {}
        if case["kind"] == "tube":
            n = s.nodes[0]
            got["rho"], got["u"] = s.out[:n].to(keep), s.out[n:].to(KEEP_U[case["precision"]])
        else:
            got["fields"] = s.out.to(keep)
        if s.ring is not None:
            got["records"] = s.ring.to(keep)
    if case["kind"] == "map":  # the outcome of a collision is read off its shell samples
        shells = np.concatenate([s.ctx.lbm_surrogate_features(k) for k in range(len(s.nodes))])
        got["shells"] = torch.from_numpy(shells).to(KEEP_U[case["precision"]])
    return got


SIZE = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}


def work(case):
    """Per step every population offset and colour record (four reals) is read
    and written once; the sampled fields are written once.  About 650 floating
    operations a node and step."""
    if case["kind"] in ("train", "predict", "gradient"):
        macs = 400 * 128 + 128 * 128 + 128 * 6
        n = case["n"]
        passes = {"predict": 2, "gradient": 6, "train": 6}[case["kind"]]
        steps = -(-n // case["batch"]) if case["kind"] == "train" else 1
        moved = 4 * (n * 393 + lbm.MLP_PARAMS * (1 if case["kind"] == "predict" else 2))
        if case["kind"] == "train":
            moved += steps * 6 * 4 * lbm.MLP_PARAMS  # weights and both moments, read and written by each update
        return {"bytes": moved, "flops": passes * n * macs}
    nodes = sum(i["p"]["nx"] * i["p"]["ny"] * i["p"]["nz"] for i in SETUPS[case["kind"]](case, 1))
    e, r = SIZE[case["precision"]], 8 if case["precision"] == "fp64" else 4
    fields = {"tube": 4, "coupled": 3}.get(case["kind"], 1)
    return {"bytes": nodes * (case["steps"] * 2 * (19 * e + 4 * r) + fields * 8), "flops": 650 * nodes * case["steps"]}


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------
C = [tuple(int(v) for v in c) for c in (
    (0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
    (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1))]
WT = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]
LEN = [1.0] * 7 + [math.sqrt(2.0)] * 12


def _at(a, c):
    """a(x + c) on the periodic lattice (last three axes z, y, x)."""
    return torch.roll(a, (-c[2], -c[1], -c[0]), (-3, -2, -1))


def _dot(c, v):
    t = 0.0
    for k in range(3):
        if c[k]:
            t = t + c[k] * v[k]
    return t


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


class Exact:
    """One instance: offsets F, colour offsets G (units of w_i rho0), spheres."""

    def __init__(self, inst, weights=None):
        p = lbm.PARAM_DEFAULTS | inst["p"]
        self.p, self.parts, self.weights = p, [], weights
        self.n3 = (p["nx"], p["ny"], p["nz"])
        self.ax = _axes(p, "cuda")
        phi, rho, u = inst["fields"]()
        shape = phi.shape
        rr, uu = rho / p["rho0"], (u * u).sum(0)
        self.F = torch.stack([rr * (1.0 + 3.0 * _dot(c, u) + 4.5 * (_dot(c, u) + 0.0 * uu) ** 2 - 1.5 * uu) - 1.0 for c in C])
        self.G = phi * (1.0 + self.F)
        self.phi, self.a, self.u = phi, torch.zeros_like(u), u.clone()
        static = torch.zeros(shape, dtype=torch.uint8, device="cuda")
        if inst.get("mask") is not None:
            static[torch.from_numpy(np.ascontiguousarray(inst["mask"])).cuda()] = 1
        if p["wall_z0"]:
            static[0] = 1
        if p["pressure_z"]:
            static[0] = static[-1] = 63
        for q in inst["parts"]:
            m = q["rho_p"] * 4.0 / 3.0 * math.pi * q["R"] ** 3
            d = dict(R=q["R"], m=m, I=0.4 * m * q["R"] ** 2, th=math.radians(q["theta_deg"]), kin=q.get("kinematic", 0),
                     q=np.array([1.0, 0, 0, 0]), Fp=np.array(p["g_particle"], float), Tp=np.zeros(3), xi=np.zeros(3),
                     xr=np.zeros(3), sub=0.0)
            for k in ("x", "v", "w"):
                d[k] = np.array(q.get(k, (0.0, 0.0, 0.0)), float)
            for k in ("Fe", "Te", "Fs", "Ts", "Fc", "Tc", "Fb"):
                d[k] = np.zeros(3)
            self.parts.append(d)
        self.static = static
        self.own = self._owners()

    def _lever(self, x):
        """Minimum-image displacements of all nodes from x, by axis."""
        return [_mi(self.ax[k] - x[k], self.n3[k]) for k in range(3)]

    def _owners(self):
        own = self.static.clone()
        for k in reversed(range(len(self.parts))):
            d = self._lever(self.parts[k]["x"])
            own[(d[0] ** 2 + d[1] ** 2 + d[2] ** 2 < self.parts[k]["R"] ** 2) & (self.static == 0)] = 2 + k
        return own

    def step(self):
        p, own, n3 = self.p, self.own, self.n3
        fluid = own == 0
        F, G = self.F, self.G
        rr = 1.0 + sum(w * f for w, f in zip(WT, F))
        j = [sum(w * c[k] * f for w, c, f in zip(WT, C, F) if c[k]) / rr for k in range(3)]
        Fi, Gi = torch.empty_like(F), torch.empty_like(G)
        acc = torch.zeros((len(self.parts), 6), dtype=F64, device="cuda")
        for i, c in enumerate(C):
            back = tuple(-v for v in c)
            so = _at(own, back)
            Fi[i], Gi[i] = _at(F[i], back), _at(G[i], back)
            z, y, x = torch.nonzero(fluid & (so != 0), as_tuple=True)
            if not len(x):
                continue
            o = so[z, y, x]
            Fo, r, ph = F[OPP[i], z, y, x], rr[z, y, x], self.phi[z, y, x]
            ca = sum(c[k] * self.a[k, z, y, x] for k in range(3)) / LEN[i]
            uw = torch.zeros((3, len(x)), dtype=F64, device="cuda")
            uw += torch.tensor(p["wall_velocity"], dtype=F64, device="cuda")[:, None] * (o == 1)
            lev = torch.zeros_like(uw)
            for k, q in enumerate(self.parts):
                mine = o == 2 + k
                d = torch.stack([_mi(t.to(F64) - 0.5 * c[b] - q["x"][b], n3[b]) for b, t in enumerate((x, y, z))])
                v = _cross(torch.tensor(q["w"], device="cuda")[:, None].expand_as(d), d)
                uw = torch.where(mine, v + torch.tensor(q["v"], device="cuda")[:, None], uw)
                lev = torch.where(mine, d, lev)
            e = 6.0 * r * _dot(c, uw)
            Fn, Gn = Fo + e, G[OPP[i], z, y, x] + ph * e
            jw = torch.stack([t[z, y, x] for t in j])
            cu = _dot(c, jw)
            rw = (p["rho_in"] if c[2] > 0 else p["rho_out"]) / p["rho0"]
            Fp = -2.0 - Fo + 2.0 * rw * (1.0 + 4.5 * cu * cu - 1.5 * (jw * jw).sum(0)) if c[2] else Fn
            press = o == 63
            Fi[i, z, y, x] = torch.where(press, Fp, Fn)
            Gi[i, z, y, x] = torch.where(press, ph * (1.0 + Fp) + ca, Gn)
            cv = torch.tensor(c, dtype=F64, device="cuda")[:, None]
            df = WT[i] * p["rho0"] * (uw * e - cv * (2.0 + 2.0 * Fo + e))
            both = torch.cat([df, _cross(lev, df)])
            for k in range(len(self.parts)):
                acc[k] += (both * (o == 2 + k)).sum(1)
        for q, s in zip(self.parts, acc.cpu().numpy()):
            q["Fe"], q["Te"] = s[:3], s[3:]
        # order parameter, also on solid nodes next to fluid
        rho = 1.0 + sum(w * f for w, f in zip(WT, Fi))
        phi = torch.where(fluid, sum(w * g for w, g in zip(WT, Gi)) / rho, 0.0)
        sw = sum(WT[i] * _at(fluid, C[i]) for i in range(1, 19))
        sp = sum(WT[i] * _at(phi, C[i]) for i in range(1, 19))
        phi = torch.where(fluid, phi, torch.where(sw > 0, sp / sw.clamp(min=1e-300), 0.0))
        g = torch.stack([3.0 * sum(WT[i] * C[i][k] * _at(phi, C[i]) for i in range(1, 19) if C[i][k]) for k in range(3)])
        self._wet(own, fluid, sw, phi, g)
        eps2 = (p["grad_eps"] or 1e-4) ** 2
        n = g / torch.sqrt((g * g).sum(0) + eps2) * fluid
        kap = 0.0
        for i in range(1, 19):
            f = _at(fluid, C[i])
            kap = kap + 3.0 * WT[i] * sum(C[i][k] * torch.where(f, _at(n[k], C[i]), n[k]) for k in range(3) if C[i][k])
        # collision (two relaxation rates on opposite pairs) with Guo forcing
        pa, pb = 0.5 * (1.0 + phi), 0.5 * (1.0 - phi)
        fo = torch.stack([-0.5 * p["sigma"] * kap * g[k] + pa * p["body_force_a"][k] + pb * p["body_force_b"][k] for k in range(3)])
        r0 = p["rho0"]
        u = torch.stack([sum(w * c[k] * f for w, c, f in zip(WT, C, Fi) if c[k]) * r0 + 0.5 * fo[k] for k in range(3)]) / (r0 * rho)
        tau = 3.0 / (((1.0 + phi) / (2.0 * r0 * p["nu_a"]) + (1.0 - phi) / (2.0 * r0 * p["nu_b"])) * r0 * rho) + 0.5
        om = 1.0 / tau
        op = 8.0 * (2.0 - om) / (8.0 - om)
        uu, uF, b = (u * u).sum(0), (u * fo).sum(0), 0.5 * p["beta"] * rho * (1.0 - phi * phi)
        Fs, Gs = torch.empty_like(F), torch.empty_like(G)
        for i, c in enumerate(C):
            cu, cF = _dot(c, u), _dot(c, fo)
            ev, od = 0.5 * (Fi[i] + Fi[OPP[i]]), 0.5 * (Fi[i] - Fi[OPP[i]])
            Fs[i] = Fi[i] - om * (ev - (rho - 1.0) - rho * (4.5 * cu * cu - 1.5 * uu)) + (1.0 - 0.5 * om) * (9.0 * cu * cF - 3.0 * uF) / r0
            Fs[i] += -op * (od - 3.0 * rho * cu) + (1.0 - 0.5 * op) * 3.0 * cF / r0
            Gs[i] = phi * (1.0 + Fs[i]) + b * _dot(c, n) / LEN[i]
        self.F, self.G = torch.where(fluid, Fs, F), torch.where(fluid, Gs, G)
        self.phi, self.a = torch.where(fluid, phi, self.phi), b * n
        self.u = u * fluid
        if self.weights is not None:
            self._surrogate(own)
        else:
            self._capillary(fluid, phi, g, eps2)
        self._dem()
        self._refill(own)

    def _wet(self, own, fluid, sw, phi, g):
        """Rotate grad(phi) at interface nodes next to a solid (Sec. V E)."""
        p = self.p
        z, y, x = torch.nonzero(fluid & (sw < 2.0 / 3.0 - 1e-9) & (phi.abs() < (p["wet_phi_max"] or 0.99)), as_tuple=True)
        if not len(x):
            return
        ws, near = torch.zeros((3, len(x)), dtype=F64, device="cuda"), torch.zeros((len(self.parts), len(x)), dtype=torch.bool, device="cuda")
        for i in range(1, 19):
            o = own[(z + C[i][2]) % self.n3[2], (y + C[i][1]) % self.n3[1], (x + C[i][0]) % self.n3[0]]
            ws -= WT[i] * torch.tensor(C[i], dtype=F64, device="cuda")[:, None] * (o == 1)
            for k in range(len(self.parts)):
                near[k] |= o == 2 + k
        ns = ws / ws.norm(dim=0).clamp(min=1e-300)
        th = torch.full((len(x),), math.radians(p["theta_wall_deg"]), dtype=F64, device="cuda")
        some = ws.norm(dim=0) > 0
        best = torch.full_like(th, math.inf)
        for k, q in enumerate(self.parts):
            d = torch.stack([_mi(t.to(F64) - q["x"][a], self.n3[a]) for a, t in enumerate((x, y, z))])
            l = d.norm(dim=0)
            take = near[k] & (l - q["R"] < best)
            best = torch.where(take, l - q["R"], best)
            ns, th = torch.where(take, d / l, ns), torch.where(take, q["th"], th)
            some |= take
        v = g[:, z, y, x]
        gm = v.norm(dim=0)
        st = -v / gm.clamp(min=1e-300)
        al = torch.acos((ns * st).sum(0).clamp(-1.0, 1.0))
        sa, ca = torch.sin(al), torch.cos(al)
        ok = some & (gm > 0) & (sa >= 1e-4)
        sa = torch.where(ok, sa, 1.0)
        up = (torch.cos(th) - torch.sin(th) * ca / sa) * ns + torch.sin(th) / sa * st
        dn = (torch.cos(th) + torch.sin(th) * ca / sa) * ns - torch.sin(th) / sa * st
        new = -gm * torch.where((up * st).sum(0) >= (dn * st).sum(0), up, dn)
        g[:, z, y, x] = torch.where(ok, new, v)

    def _corners(self, X, fluid):
        """Indices, trilinear weights over fluid corners of points X [3, m]."""
        b = torch.floor(X)
        f, out = X - b, []
        for dz in range(2):
            for dy in range(2):
                for dx in range(2):
                    at = tuple((b[k].long() + d) % self.n3[k] for k, d in ((2, dz), (1, dy), (0, dx)))
                    w = 1.0
                    for k, d in ((0, dx), (1, dy), (2, dz)):
                        w = w * (f[k] if d else 1.0 - f[k])
                    out.append((at, w * fluid[at]))
        return out

    def _capillary(self, fluid, phi, g, eps2):
        p = self.p
        da = math.radians(2.0)
        al = ((torch.arange(90, dtype=F64, device="cuda") + 0.5) * da)[:, None].expand(90, 180).reshape(-1)
        vp = (torch.arange(180, dtype=F64, device="cuda") * da)[None, :].expand(90, 180).reshape(-1)
        ns = torch.stack([torch.sin(al) * torch.cos(vp), torch.sin(al) * torch.sin(vp), torch.cos(al)])
        norm = p["cap_norm"] or 3.0 * (1.0 + math.sqrt(2.0)) / 18.0 * p["beta"]
        for q in self.parts:
            cor = self._corners(torch.tensor(q["x"], device="cuda")[:, None] + q["R"] * ns, fluid)
            ws = sum(w for _, w in cor)
            some, den = ws > 0, ws.clamp(min=1e-300)
            ph = sum(w * phi[at] for at, w in cor) / den
            gr = torch.stack([sum(w * g[k][at] for at, w in cor) / den for k in range(3)])
            nn = gr / torch.sqrt((gr * gr).sum(0) + eps2)
            dA = q["R"] ** 2 * torch.sin(al) * da * da
            dF = norm * p["sigma"] * (1.0 - ph * ph) * dA * _cross(_cross(nn, ns), nn) * (some & (ph.abs() < 1.0))
            q["Fs"], q["Ts"] = dF.sum(1).cpu().numpy(), _cross(q["R"] * ns, dF).sum(1).cpu().numpy()
            if any(p["buoyancy_a"]):
                area = float((dA * some).sum())
                t = 2.0 * float(((0.5 * (1.0 + ph)).clamp(0.0, 1.0) * dA * some).sum()) / area - 1.0 if area > 0 else -1.0
                q["sub"] = (1.0 + t) ** 2 * (2.0 - t) / 4.0
                q["Fb"] = 4.0 / 3.0 * math.pi * q["R"] ** 3 * q["sub"] * np.array(p["buoyancy_a"], float)

    def shells(self, own):
        """The surrogate's inputs of every sphere [n, 387]."""
        p, k = self.p, torch.arange(96, dtype=F64, device="cuda")
        ez = 1.0 - (2.0 * k + 1.0) / 96.0
        az = k * (math.pi * (3.0 - math.sqrt(5.0)))
        e = torch.stack([torch.sqrt(1.0 - ez * ez) * torch.cos(az), torch.sqrt(1.0 - ez * ez) * torch.sin(az), ez])
        rows, fluid = [], own == 0
        for q in self.parts:
            lev = (q["R"] + (p["surrogate_shell_gap"] or 2.0)) * e
            X = torch.tensor(q["x"], device="cuda")[:, None] + lev
            inside = ((X[2] >= 0.0) & (X[2] < self.n3[2])) if p["wall_z0"] else torch.ones_like(ez, dtype=torch.bool)
            X = torch.stack([X[a] - self.n3[a] * torch.floor(X[a] / self.n3[a]) for a in range(3)])
            cor = self._corners(X, fluid)
            ws = sum(w for _, w in cor)
            ok, den = (ws > 0) & inside, ws.clamp(min=1e-300)
            w3 = torch.tensor(q["w"], device="cuda")[:, None].expand_as(lev)
            us = torch.tensor(q["v"], device="cuda")[:, None] + _cross(w3, lev)
            cols = [sum(w * self.phi[at] for at, w in cor) / den]
            cols += [(sum(w * self.u[a][at] for at, w in cor) / den - us[a]) / (p["surrogate_u_ref"] or 1e-3) for a in range(3)]
            row = (torch.stack(cols, 1) * ok[:, None]).reshape(-1)
            tail = torch.tensor([math.cos(q["th"]), math.sin(q["th"]), q["R"] / (p["surrogate_r_ref"] or 8.0)], dtype=F64, device="cuda")
            rows.append(torch.cat([row, tail]))
        return torch.stack(rows)

    def _surrogate(self, own):
        y = _network(self.weights, self.shells(own).float())[0].cpu().numpy()
        for q, o in zip(self.parts, y):
            s = self.p["sigma"] * q["R"]
            q["Fe"], q["Te"], q["Fs"], q["Ts"] = s * o[:3], s * q["R"] * o[3:], np.zeros(3), np.zeros(3)

    def _dem(self):
        """Substrate contacts (the spheres start clear of one another) and velocity Verlet."""
        p = self.p

        def spring(xi, n, v, k, gam, cap):
            xi = xi - np.dot(xi, n) * n
            F0 = -k * xi - gam * v
            m = np.linalg.norm(F0)
            if m <= cap:
                return F0, xi + v
            F = cap * F0 / m
            return F, -(F + gam * v) / k if k > 0 else np.zeros(3)

        n = np.array([0.0, 0.0, 1.0])
        for q in self.parts:
            acc, alp = (np.zeros(3), np.zeros(3)) if q["kin"] else (q["Fp"] / q["m"], q["Tp"] / q["I"])
            xn, vp, wp = q["x"] + q["v"] + 0.5 * acc, q["v"] + acc, q["w"] + alp
            q["Fc"], q["Tc"] = np.zeros(3), np.zeros(3)
            Rc = q["R"] + p["delta_R"]
            delta = Rc - (xn[2] - 0.5)
            if p["wall_z0"] and delta > 0.0:
                arm = -(Rc - 0.5 * delta) * n
                vr = vp + np.cross(wp, arm) - np.array(p["wall_velocity"], float)
                Fn = p["kn"] * delta - p["gn"] * np.dot(vr, n)
                Ft, q["xi"] = spring(q["xi"], n, vr - np.dot(vr, n) * n, p["kt"], p["gt"], p["mu_s"] * abs(Fn))
                Fr, q["xr"] = spring(q["xr"], n, -Rc * np.cross(wp, n), p["kr"], p["gr"], p["mu_r"] * abs(Fn))
                q["Fc"], q["Tc"] = Fn * n + Ft, np.cross(arm, Ft) - Rc * np.cross(n, Fr)
            else:
                q["xi"], q["xr"] = np.zeros(3), np.zeros(3)
            F = q["Fc"] + np.array(p["g_particle"], float) + q["Fe"] + q["Fs"] + q["Fb"]
            T = q["Tc"] + q["Te"] + q["Ts"]
            w0 = q["w"]
            if not q["kin"]:
                q["v"], q["w"] = q["v"] + 0.5 * (q["Fp"] + F) / q["m"], q["w"] + 0.5 * (q["Tp"] + T) / q["I"]
            wm = 0.5 * (w0 + q["w"])
            a = np.linalg.norm(wm)
            if a > 0.0:
                d, s = math.cos(0.5 * a), math.sin(0.5 * a) / a * wm
                r = np.concatenate([[d * q["q"][0] - s @ q["q"][1:]], d * q["q"][1:] + q["q"][0] * s + np.cross(s, q["q"][1:])])
                q["q"] = r / np.linalg.norm(r)
            q["x"], q["Fp"], q["Tp"] = xn - np.array(self.n3) * np.floor(xn / np.array(self.n3)), F, T

    def _refill(self, before):
        self.own = self._owners()
        z, y, x = torch.nonzero((self.own == 0) & (before >= 2) & (before < 63), as_tuple=True)
        if not len(x):
            return
        good = (self.own == 0) & (before == 0)
        rr, F = 1.0 + sum(w * f for w, f in zip(WT, self.F)), self.F.clone()
        for zz, yy, xx in zip(z.tolist(), y.tolist(), x.tolist()):
            for hop in (1, 2):
                s = [((zz + hop * c[2]) % self.n3[2], (yy + hop * c[1]) % self.n3[1], (xx + hop * c[0]) % self.n3[0]) for c in C[1:]]
                s = [t for t in s if bool(good[t])]
                if s:
                    break
            r = sum(float(rr[t]) for t in s) / len(s) if s else 1.0
            d = sum(float(rr[t] * self.phi[t]) for t in s) / len(s) if s else -1.0
            q = self.parts[int(before[zz, yy, xx]) - 2]
            arm = np.array([v - n * math.floor(v / n + 0.5) for v, n in zip(np.array([xx, yy, zz]) - q["x"], self.n3)])
            u = q["v"] + np.cross(q["w"], arm)
            e = [1.0 + 3.0 * np.dot(c, u) + 4.5 * np.dot(c, u) ** 2 - 1.5 * np.dot(u, u) for c in C]
            F[:, zz, yy, xx] = torch.tensor([r * v - 1.0 for v in e], dtype=F64, device="cuda")
            self.phi[zz, yy, xx] = d / r
            self.G[:, zz, yy, xx] = d / r * (1.0 + F[:, zz, yy, xx])
            self.a[:, zz, yy, xx] = 0.0
        self.F = F

    def records(self):
        return np.array([np.concatenate([q["Fe"], q["Te"], q["Fs"], q["Ts"], q["Fc"], q["Tc"], q["x"], q["v"], q["w"], q["q"],
                                         [q["m"], q["sub"]], q["Fb"]]) for q in self.parts])

    def fields(self):
        fluid = self.own == 0
        r = self.p["rho0"] * (1.0 + sum(w * f for w, f in zip(WT, self.F))) * fluid
        d = self.p["rho0"] * sum(w * g for w, g in zip(WT, self.G)) * fluid
        return 0.5 * (r + d), 0.5 * (r - d), torch.where(fluid, d / torch.where(fluid, r, 1.0), 0.0)


def _b(t):
    """The value as a BF16 operand of the network's products holds it."""
    return t.to(torch.bfloat16).to(F64)


def _split(th):
    at = np.cumsum([0, 128 * 400, 128, 128 * 128, 128, 6 * 128, 6])
    shape = [(128, 400), (128,), (128, 128), (128,), (6, 128), (6,)]
    return [th[a:b].reshape(s) for a, b, s in zip(at[:-1], at[1:], shape)]


def _network(th, X):
    """Outputs and hidden layers for inputs X [n, 387] (BF16 operands, 64-bit sums)."""
    W1, b1, W2, b2, W3, b3 = _split(th)
    x = _b(torch.nn.functional.pad(X, (0, 13)))
    h1 = _b(torch.tanh(x @ _b(W1).T + b1).float())
    h2 = _b(torch.tanh(h1 @ _b(W2).T + b2).float())
    return h2 @ _b(W3).T + b3, h2, h1, x


def _gradient(th, X, Y):
    W1, b1, W2, b2, W3, b3 = _split(th)
    y, h2, h1, x = _network(th, X)
    d = 2.0 * (y - Y.double()) / y.numel()
    dy = _b(d.float())
    z2 = _b((dy @ _b(W3) * (1.0 - h2 * h2)).float())
    z1 = _b((z2 @ _b(W2) * (1.0 - h1 * h1)).float())
    parts = [z1.T @ x, z1.sum(0), z2.T @ h1, z2.sum(0), dy.T @ h2, d.sum(0)]
    return torch.cat([t.reshape(-1) for t in parts]), float(((y - Y.double()) ** 2).mean())


def _order(n, state):
    """Fisher-Yates order drawn from SplitMix64 (published constants)."""
    perm, M = list(range(n)), (1 << 64) - 1
    for i in range(n - 1, 0, -1):
        state = (state + 0x9E3779B97F4A7C15) & M
        v = state
        v = ((v ^ (v >> 30)) * 0xBF58476D1CE4E5B9) & M
        v = ((v ^ (v >> 27)) * 0x94D049BB133111EB) & M
        k = (v ^ (v >> 31)) % (i + 1)
        perm[i], perm[k] = perm[k], perm[i]
    return perm


def exact(case, seed):
    if case["kind"] in ("train", "predict", "gradient"):
        th = torch.from_numpy(_weights(seed)).cuda().double()
        X, Y = (torch.from_numpy(t).cuda() for t in _samples(case["n"], seed))
        if case["kind"] == "predict":
            return _network(th, X)[0]
        if case["kind"] == "gradient":
            return _gradient(th, X, Y)
        m, v, losses = torch.zeros_like(th), torch.zeros_like(th), []
        order = torch.tensor(_order(case["n"], seed), device="cuda")
        for t, at in enumerate(order.split(case["batch"]), 1):
            g, loss = _gradient(th, X[at], Y[at])
            losses.append(loss)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            th = th - 1e-3 * (m / (1.0 - 0.9 ** t)) / (torch.sqrt(v / (1.0 - 0.999 ** t)) + 1e-8)
        return th, sum(losses) / len(losses)
    fields, u, records, shells = [], [], [], []
    weights = torch.from_numpy(_weights(seed)).cuda().double() if case["kind"] == "coarse" else None
    for inst in SETUPS[case["kind"]](case, seed):
        s, recs = Exact(inst, weights), []
        for _ in range(case["steps"]):
            s.step()
            recs.append(s.records())
        ra, rb, phi = s.fields()
        fields += {"tube": [ra], "coupled": [ra, rb, phi]}.get(case["kind"], [phi])
        u.append(s.u)
        records.append(recs)
        if case["kind"] == "map":
            shells.append(s.shells(s.own))
    flat = torch.cat([f.reshape(-1) for f in fields])
    got = {"rho": flat, "u": u[0].reshape(-1)} if case["kind"] == "tube" else {"fields": flat}
    if records[0][0].size:
        got["records"] = np.ascontiguousarray(np.concatenate([np.array(r) for r in records], axis=1))
    if shells:
        got["shells"] = torch.cat(shells)
    return got
