"""Workloads for timing the library through its public entry points.

A case is a dict of plain values; ``prepare`` builds what a program holds before the call (the
simulation in its stirred state, the trained network, the logged rows), ``run`` is one pass as a
program makes it, ``exact`` the same outputs in 64 bits from plain torch, where that is feasible.

Kinds of case, and the use each stands for:

haptic      One displayed frame of an interactive scene: the 1 kHz haptic loop sets the grabbed
            cube's pose, advances one substep and reads the wrench, 16 times; then the frame's
            particle state is read.  The dam break with a grabbed cube, from a seeded velocity
            field.  Small: launches, latency and the serial chains of single particles count.
            ``low_latency``: the opt-in passes for such scenes.
stirring    The stirring tank under its paddle's path: one update cycle of substeps, then the
            wrenches of the cycle and the state, as a logging run does.
coupled     The same for the coupled scene (random-walk probe, soft cube), up to the
            1.16 M-particle one, from its stirred state; optionally with volume-based boundaries
            or the Tait equation of state, or with the low-latency passes.
batch       Many small stirring scenes advanced together (training episodes), then every
            scene's wrench and state.
isosurface  The fluid surface of a stirred scene for display: corner field and triangles.
tick        The learned surrogate between two update cycles: the cycle's anchor, then 16 ticks at
            1 kHz, each a pose in and a wrench out.  The smallest calls there are.
train       Minibatch Adam steps of the surrogate, then its parameters (as at a checkpoint).
infer       Offline evaluation of the surrogate: inputs of logged rows, then their predictions.
sort        The allocation-free spatial hash of a caller's own particles (keys, order, ranges).

Sizes are those of the repository's scenes, benchmark forms and tests.
"""
import math

import numpy as np
import torch

from paper_2511_15908_gb300 import scenes, sph

DEV = torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")


def listed():
    return [
        # the smallest calls: a haptic tick answered by the network
        {"name": "tick_cycle", "kind": "tick", "n_side": 16, "ticks": 16},
        # the 12k-particle dam break with a grabbed cube, a frame of 16 haptic cycles
        {"name": "haptic_dam_break", "kind": "haptic", "n_side": 16, "cycles": 16, "low_latency": False},
        # the same with the passes made for small scenes
        {"name": "haptic_dam_break_fast", "kind": "haptic", "n_side": 16, "cycles": 16, "low_latency": True},
        # an interactive scene with a soft body, between the small and the chip-filling ones
        {"name": "interactive_60k_tait", "kind": "coupled", "cols_x": 60, "cols_y": 40, "n_fluid": 60_000,
         "probe_r": 0.04, "soft_n": 8, "substeps": 16, "flags": scenes.FLAG_TAIT | sph.FLAG_LOW_LATENCY},
        # the 250k stirring tank, one 60 Hz update cycle of 32 substeps
        {"name": "stirring_250k", "kind": "stirring", "cols": 125, "n_fluid": 250_000, "substeps": 32},
        # an odd size with volume-based boundaries
        {"name": "volume_217k", "kind": "coupled", "cols_x": 97, "cols_y": 89, "n_fluid": 217_373,
         "probe_r": 0.06, "soft_n": 12, "substeps": 32, "flags": scenes.FLAG_VOLUME_BOUNDARY},
        # the headline scene: 1 M fluid particles, 100 substeps between two logged states
        {"name": "coupled_1m", "kind": "coupled", "cols_x": 200, "cols_y": 100, "n_fluid": 1_000_000,
         "probe_r": 0.0964, "soft_n": 24, "substeps": 100, "flags": 0},
        # 64 compact scenes of 0.5k to 2k fluid particles
        {"name": "batch_64", "kind": "batch", "scenes": 64, "lo": 500, "hi": 2000, "substeps": 64},
        # the surface of a stirred 250k scene
        {"name": "isosurface_250k", "kind": "isosurface", "cols_x": 100, "cols_y": 100, "n_fluid": 250_000,
         "cube_over_h": 1.0},
        # eight Adam steps at the benchmark's minibatch
        {"name": "train_1024", "kind": "train", "batch": 1024, "steps": 8},
        # the offline evaluation's batch
        {"name": "infer_4096", "kind": "infer", "rows": 4096},
        # a caller's own particles, near the call's largest count
        {"name": "sort_200k", "kind": "sort", "n": 200_003, "cells": 50},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["haptic", "haptic", "stirring", "coupled", "coupled", "batch", "isosurface", "tick", "train",
                       "infer", "sort"])
    if kind == "haptic":
        return {"kind": kind, "n_side": rng.randint(8, 16), "cycles": rng.randint(4, 24),
                "low_latency": rng.random() < 0.5}
    if kind == "stirring":
        cols = _log_int(rng, 44, 125)
        return {"kind": kind, "cols": cols, "n_fluid": cols * cols * rng.randint(8, 16) - rng.randint(0, 99),
                "substeps": rng.randint(8, 40)}
    if kind == "coupled":
        flags = rng.choice([0, 0, scenes.FLAG_VOLUME_BOUNDARY, scenes.FLAG_TAIT, sph.FLAG_LOW_LATENCY])
        big = 90 if flags & sph.FLAG_LOW_LATENCY else 200
        cx, cy = _log_int(rng, 50, big), _log_int(rng, 40, 100)
        return {"kind": kind, "cols_x": cx, "cols_y": cy, "n_fluid": cx * cy * rng.randint(20, 45) - rng.randint(0, 99),
                "probe_r": round(rng.uniform(0.03, 0.06), 4), "soft_n": rng.randint(6, 12),
                "substeps": rng.randint(8, 40), "flags": flags}
    if kind == "batch":
        lo = _log_int(rng, 200, 2000)
        return {"kind": kind, "scenes": _log_int(rng, 16, 96), "lo": lo, "hi": 4 * lo, "substeps": rng.randint(16, 48)}
    if kind == "isosurface":
        cx, cy = _log_int(rng, 50, 160), _log_int(rng, 40, 100)
        return {"kind": kind, "cols_x": cx, "cols_y": cy, "n_fluid": cx * cy * rng.randint(15, 30) - rng.randint(0, 99),
                "cube_over_h": round(rng.uniform(0.8, 2.0), 3)}
    if kind == "tick":
        return {"kind": kind, "n_side": rng.randint(8, 16), "ticks": rng.randint(8, 32)}
    if kind == "train":
        return {"kind": kind, "batch": _log_int(rng, 64, 4096), "steps": rng.randint(2, 8)}
    if kind == "infer":
        return {"kind": kind, "rows": _log_int(rng, 16, 16384)}
    return {"kind": kind, "n": _log_int(rng, 500, 262144), "cells": rng.randint(16, 60)}


# ------------------------------------------------------------------------------ inputs

def _there_and_back(path):
    """A path that can be walked forever without a jump: forward, then backward."""
    back = path[::-1].copy()
    back[:, 7:] *= -1.0
    return np.ascontiguousarray(np.concatenate([path, back]))


def _haptic_scene(case, seed):
    side = case["n_side"] * 0.02              # the cube starts beside the fluid, within its reach
    sc = scenes.dam_break(seed=seed, n_side=case["n_side"], grab=True, n_substeps=1500,
                          cube_pos=(side + 0.06, 0.5 * side, 0.1))
    sc = scenes.with_velocity_noise(sc, seed=seed + 1, sigma=0.1)
    sc.trajectory[:, 10:13] *= 0.0            # the cube is carried without spinning
    if case.get("low_latency"):
        sc.params["flags"] |= sph.FLAG_LOW_LATENCY
    return sc


def _coupled_scene(case, seed, flags):
    cx, cy, s = case["cols_x"], case["cols_y"], 0.01
    depth = case["n_fluid"] / (cx * cy) * s
    sc = scenes.coupled(seed=seed, n_fluid=case["n_fluid"], cols=(cx, cy),
                        tank=(cx * s, cy * s, max(0.4, round(1.2 * depth, 2))), n_substeps=3000,
                        probe_r=case.get("probe_r", 0.04), soft_n=case.get("soft_n", 8))
    sc.trajectory = _there_and_back(sc.trajectory)
    sc.params["flags"] |= flags
    return sc


def _stirring_scene(seed, n_fluid, cols, tank_z=0.5, paddle=(0.02, 0.2, 0.3)):
    return scenes.stirring_tank(seed=seed, n_fluid=n_fluid, cols=(cols, cols),
                                tank=(cols * 0.008, cols * 0.008, tank_z), n_substeps=6000, paddle=paddle)


def _mlp_rows(n, seed):
    """Logged rows as the surrogate sees them: tick pose and velocity, anchor descriptor (pose,
    velocity, 64 cells of density and velocity, some of them empty), time since the anchor."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, device=DEV, generator=g)

    q = normal(n, 4)
    q = q / q.norm(dim=1, keepdim=True)
    x = 0.25 + 0.05 * normal(n, 3)
    v, w = 0.2 * normal(n, 3), 0.5 * normal(n, 3)
    rho = 1000.0 + 3.0 * normal(n, 64, 1)
    cells = torch.cat([rho, 0.15 * normal(n, 64, 3)], 2)
    cells = cells * (torch.rand(n, 64, 1, device=DEV, generator=g) > 0.2)
    anchors = torch.cat([x, q, v, w, cells.reshape(n, 256)], 1).contiguous()
    tau = 1e-3 * torch.randint(0, 16, (n,), device=DEV, generator=g).float()
    v2 = v + 0.05 * normal(n, 3)
    ticks = torch.cat([x + v * tau[:, None], q, v2, w + 0.1 * normal(n, 3)], 1).contiguous()
    return ticks, anchors, tau


SCENE = dict(h=0.02, k=64.0, rho0=1000.0, nu=1e-3, g=(0.0, 0.0, -9.81), dt=1e-3, lo=(-0.06,) * 3, hi=(0.56, 0.56, 0.75),
             cell=0.02002, flags=1, visc_eps=0.01, spring_zeta=0.1)


def _train_rows(case, seed):
    """Minibatches of standardisable inputs and of targets that depend on them smoothly."""
    n = case["batch"]
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    mix = torch.randn(269, 24, device=DEV, generator=g) / math.sqrt(269)
    out = torch.randn(24, 6, device=DEV, generator=g) / math.sqrt(24)
    xs = [torch.randn(n, 269, device=DEV, generator=g) * 0.7 + 0.1 for _ in range(8)]
    ys = [0.3 * (torch.tanh(2.0 * x @ mix) @ out + 0.02 * torch.randn(n, 6, device=DEV, generator=g)) for x in xs]
    norm = np.concatenate([np.full(269, 0.1), np.full(269, 0.7), np.zeros(6), np.full(6, 0.25)]).astype(np.float32)
    return xs, ys, norm


TRAIN_LR = 3e-4


# ------------------------------------------------------------------------------- cases

def prepare(case, seed):
    kind = case["kind"]
    if kind == "haptic":
        sc = _haptic_scene(case, seed)
        path = _there_and_back(sc.trajectory)
        sc.trajectory = None                  # the device, not a stored path, gives the pose
        sc.bodies[1].pose = path[0, :7].copy()
        sim = sph.Simulation(sc)
        return {"kind": kind, "sim": sim, "body": sim.body_ids[1], "path": path, "at": 0, "cycles": case["cycles"]}
    if kind in ("stirring", "coupled"):
        if kind == "stirring":
            sc = _stirring_scene(seed, case["n_fluid"], case["cols"])
        else:
            sc = _coupled_scene(case, seed, case["flags"])
        sim = sph.Simulation(sc)
        sim.step(200)                         # from the seeded fill to the stirred state
        return {"kind": kind, "sim": sim, "substeps": case["substeps"]}
    if kind == "batch":
        rng = np.random.default_rng(1)        # the sizes belong to the case, the jitter to the seed
        counts = np.exp(rng.uniform(np.log(case["lo"]), np.log(case["hi"]), case["scenes"])).astype(int)
        sims = []
        for i, n in enumerate(counts):
            side = max(int(math.ceil(math.sqrt(n / 16.0))), 12)
            paddle = (0.02, min(0.2, 0.25 * side * 0.008), 0.15)
            sims.append(sph.Simulation(_stirring_scene(1000 * seed + i, int(n), side, 0.2, paddle)))
        batch = sph.Batch(sims)
        batch.configure(0)                    # one launch per phase: what its tuner picks for such sets
        batch.step(20)
        batch.sync()
        return {"kind": kind, "sims": sims, "batch": batch, "substeps": case["substeps"]}
    if kind == "isosurface":
        sim = sph.Simulation(_coupled_scene(case, seed, 0))
        sim.step(60)
        sim.sync()
        p = sim.scene.params
        cube = float(np.float32(case["cube_over_h"] * p["h"]))
        dims, origin = sph.iso_grid(p, cube)
        vertices = torch.zeros(16 * case["cols_x"] * case["cols_y"], 3, 3, device=DEV)   # a renderer's buffer
        return {"kind": kind, "sim": sim, "cube": cube, "dims": dims, "origin": origin, "iso": 0.5 * p["rho0"],
                "vertices": vertices}
    if kind == "tick":
        sc = _haptic_scene(case, seed)
        sc.trajectory = _there_and_back(sc.trajectory)
        sim = sph.Simulation(sc)
        sim.step(20)
        sim.sync()
        model = sph.Surrogate(max_batch=1024)
        norm = np.concatenate([np.zeros(269), np.full(269, 0.5), np.zeros(6), np.full(6, 0.02)]).astype(np.float32)
        model.set_params(scenes.mlp_init_params(seed), norm)
        return {"kind": kind, "sim": sim, "model": model, "path": sc.trajectory[20:20 + case["ticks"]]}
    if kind == "train":
        xs, ys, norm = _train_rows(case, seed)
        model = sph.Surrogate(max_batch=case["batch"])
        model.set_params(scenes.mlp_init_params(seed), norm)
        return {"kind": kind, "model": model, "xs": xs, "ys": ys, "steps": case["steps"]}
    if kind == "infer":
        ticks, anchors, tau = _mlp_rows(case["rows"], seed)
        model = sph.Surrogate(max_batch=case["rows"])
        norm = np.concatenate([np.zeros(269), np.full(269, 0.5), np.zeros(6), np.full(6, 0.02)]).astype(np.float32)
        model.set_params(scenes.mlp_init_params(seed), norm)
        model.set_scene(SCENE)
        return {"kind": kind, "model": model, "ticks": ticks, "anchors": anchors, "tau": tau}
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    x = torch.rand(case["n"], 4, device=DEV, generator=g)
    x[:, 2] *= 0.5                            # the fluid fills the lower half
    edge = 1.0 / case["cells"]
    params = dict(SCENE, h=edge, cell=edge, lo=(0.0,) * 3, hi=(1.0,) * 3)
    return {"kind": "sort", "x": x.contiguous(), "params": params}


def _reported(read):
    """A read of the run's results; a latched out-of-domain report (a splash clamped into the
    border cells) is cleared by the read that raises it."""
    try:
        return read()
    except sph.SphError as e:
        if e.status != sph.ERR_DOMAIN:
            raise
        return read()


def run(s):
    kind = s["kind"]
    if kind == "haptic":
        sim, path, wrench = s["sim"], s["path"], np.zeros((s["cycles"], 6))
        for j in range(s["cycles"]):
            row = path[s["at"] % len(path)]
            s["at"] += 1
            try:
                sim.haptic_cycle(s["body"], row[:7], row[7:], out=wrench[j])
            except sph.SphError as e:
                if e.status != sph.ERR_DOMAIN:
                    raise
        st = _reported(sim.state)
        return {"wrench": wrench, "x": st["x"], "v": st["v"], "rho": st["rho"]}
    if kind in ("stirring", "coupled"):
        sim = s["sim"]
        sim.step(s["substeps"])
        log = _reported(lambda: sim.wrench_log(s["substeps"]))
        st = sim.state()
        return {"wrench": log, "x": st["x"], "v": st["v"], "rho": st["rho"]}
    if kind == "batch":
        s["batch"].step(s["substeps"])
        s["batch"].sync()
        wrench = np.stack([_reported(sim.grab_wrench) for sim in s["sims"]])
        st = [sim.state() for sim in s["sims"]]
        return {"wrench": wrench, **{k: np.concatenate([t[k] for t in st]) for k in ("x", "v", "rho")}}
    if kind == "isosurface":
        field, vertices = s["sim"].iso_field(s["cube"]), s["vertices"]
        tris = sph.iso_polygonize(field, s["dims"], s["origin"], s["cube"], s["iso"], max_tris=vertices.shape[0])
        vertices[:tris.shape[0]].copy_(tris)
        vertices[tris.shape[0]:].zero_()
        return {"field": field, "triangles": vertices, "count": tris.shape[0]}
    if kind == "tick":
        model, out = s["model"], np.zeros((len(s["path"]), 6))
        model.anchor(s["sim"])
        for j, row in enumerate(s["path"]):
            model.tick(row, 1e-3 * j, out=out[j])
        return out
    if kind == "train":
        loss = None
        for j in range(s["steps"]):
            loss = s["model"].train_step(s["xs"][j], s["ys"][j], TRAIN_LR, want_loss=j == s["steps"] - 1)
        return {"params": s["model"].get_params(), "loss": float(np.float32(loss))}
    if kind == "infer":
        x = s["model"].features(s["ticks"], s["anchors"], s["tau"])
        return {"x": x, "y": s["model"].forward(x)}
    keys, order, start = sph.cell_sort_noalloc(s["params"], s["x"])
    return {"keys": keys, "order": order, "start": start}


def _particles(case):
    kind = case["kind"]
    if kind in ("haptic", "tick"):
        return case["n_side"] ** 3 + 8000
    if kind == "batch":
        return int(case["scenes"] * (math.sqrt(case["lo"] * case["hi"]) + 4000))
    if kind == "stirring":
        return int(case["n_fluid"] + 6.2 * case["cols"] ** 2 + 18750)
    cx, cy = case["cols_x"], case["cols_y"]
    walls = 2 * cx * cy + 4 * (cx + cy) * max(40, int(1.2 * case["n_fluid"] / (cx * cy)))
    probe = 4.19 * (case.get("probe_r", 0.04) / 0.005) ** 3
    return int(case["n_fluid"] + walls + probe + case.get("soft_n", 8) ** 3)


def work(case):
    """Bytes: every input read once and every output written once per substep (position,
    velocity and the two density values of a particle, 32 + 40 bytes; once more 28 bytes for the
    state handed out).  Flops: 15 per density pair and 50 per force pair, about 34 and 26 of
    them per particle; a network row costs two per weight forward and four backward."""
    kind, weights = case["kind"], 68_096
    if kind in ("haptic", "stirring", "coupled", "batch"):
        n, steps = _particles(case), case.get("substeps", case.get("cycles"))
        return {"bytes": n * (72.0 * steps + 28.0), "flops": n * steps * (34 * 15.0 + 26 * 50.0)}
    if kind == "isosurface":
        n = _particles(case)
        corners = n / case["cube_over_h"] ** 3
        return {"bytes": 32.0 * n + 8.0 * corners, "flops": 33 * 15.0 * corners}
    if kind == "tick":
        return {"bytes": 4.0 * weights * case["ticks"], "flops": 2.0 * weights * case["ticks"]}
    if kind == "train":
        rows = case["batch"] * case["steps"]
        return {"bytes": 4.0 * 275 * rows + 24.0 * weights * case["steps"], "flops": 6.0 * weights * rows}
    if kind == "infer":
        return {"bytes": 4.0 * case["rows"] * (13 + 269 + 1 + 269 + 6) + 2.0 * weights, "flops": 2.0 * weights * case["rows"]}
    return {"bytes": (16.0 + 8.0) * case["n"] + 4.0 * case["cells"] ** 3, "flops": 9.0 * case["n"]}


# ------------------------------------------------------------------------- in 64 bits

def exact(case, seed):
    if case["kind"] == "haptic":
        return _exact_haptic(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "infer":
        return _exact_infer(case, seed)
    return None       # long runs of large scenes from a stirred state; whole numbers


def _pairwise(x, h, fn, rows=1024):
    """fn(row indices, column indices, d = x_j - x_i, r) summed over neighbours, by row blocks."""
    for a in range(0, x.shape[0], rows):
        xi = x[a:a + rows]
        near = torch.cdist(xi, x, compute_mode="donot_use_mm_for_euclid_dist") < 2.0 * h
        i, j = near.nonzero(as_tuple=True)
        d = x[j] - xi[i]
        fn(i + a, j, d, d.square().sum(1).sqrt())


def _exact_haptic(case, seed):
    """The substep by its definition: all pairs, every operation in 64 bits."""
    sc = _haptic_scene(case, seed)
    f64 = dict(dtype=torch.float64, device=DEV)
    path = _there_and_back(sc.trajectory)
    walls, cube = sc.bodies
    f32 = {k: float(np.float32(sc.params[k])) for k in ("h", "k", "rho0", "nu", "dt", "visc_eps")}
    h, rho0, dt = f32["h"], f32["rho0"], f32["dt"]
    grav = torch.tensor(np.array(sc.params["g"], np.float32).astype(np.float64), **f64)
    nf, nw, n = sc.n_fluid, walls.n, sc.n_total
    x = torch.zeros(n, 3, **f64)
    v = torch.zeros(n, 3, **f64)
    x[:nf] = torch.tensor(sc.fluid_x, **f64)
    v[:nf] = torch.tensor(sc.fluid_v, **f64)
    x[nf:nf + nw] = torch.tensor(walls.xyz, **f64)
    local = torch.tensor(cube.xyz, **f64)
    m = torch.empty(n, **f64)
    for lo, hi, s in ((0, nf, sc.fluid_spacing), (nf, nf + nw, walls.spacing), (nf + nw, n, cube.spacing)):
        m[lo:hi] = float(np.float32(rho0) * np.float32(s) ** 3)
    owner = torch.zeros(n, dtype=torch.int64, device=DEV)
    owner[nf:nf + nw] = 1
    owner[nf + nw:] = 2
    alpha = 3.0 / (2.0 * math.pi * h ** 3)
    wrench = torch.zeros(case["cycles"], 6, **f64)
    rho = None
    for step in range(case["cycles"]):
        row = torch.tensor(path[step % len(path)].astype(np.float64), **f64)
        t, vel, spin = row[:3], row[7:10], row[10:13]
        w, a, b, c = (float(u) for u in row[3:7])
        rot = torch.tensor([[1 - 2 * (b * b + c * c), 2 * (a * b - w * c), 2 * (a * c + w * b)],
                            [2 * (a * b + w * c), 1 - 2 * (a * a + c * c), 2 * (b * c - w * a)],
                            [2 * (a * c - w * b), 2 * (b * c + w * a), 1 - 2 * (a * a + b * b)]], **f64)
        arm = local @ rot.T
        x[nf + nw:] = arm + t
        v[nf + nw:] = vel + torch.linalg.cross(spin.expand_as(arm), arm)
        rho = torch.zeros(n, **f64)

        def density(i, j, d, r):
            q = r / h
            wq = ((2 - q).clamp(min=0) ** 3 - 4 * (1 - q).clamp(min=0) ** 3) / 6
            rho.index_add_(0, i, alpha * m[j] * wq)

        _pairwise(x, h, density)
        p = (f32["k"] * (rho - rho0)).clamp(min=0)
        pr = p / rho.square()
        acc = torch.zeros(n, 3, **f64)

        def force(i, j, d, r):
            keep = (r > 0) & ~((owner[i] == owner[j]) & (owner[i] > 0))
            i, j, d, r = i[keep], j[keep], d[keep], r[keep]
            q = r / h
            g = torch.where(q < 1, -2 * q + 1.5 * q * q, -0.5 * (2 - q) ** 2) / q * (alpha / h ** 2)
            vx = -((v[i] - v[j]) * d).sum(1)
            visc = 20 * f32["nu"] * vx / ((rho[i] + rho[j]) * (r * r + f32["visc_eps"] * h * h))
            acc.index_add_(0, i, (m[j] * (pr[i] + pr[j] - visc) * g)[:, None] * d)

        _pairwise(x, h, force)
        f = m[nf + nw:, None] * acc[nf + nw:]
        wrench[step, :3] = f.sum(0)
        wrench[step, 3:] = torch.linalg.cross(x[nf + nw:] - t, f).sum(0)
        v[:nf] += (acc[:nf] + grav) * dt
        x[:nf] += v[:nf] * dt
    return {"wrench": wrench, "x": x, "v": v, "rho": rho}


def _mlp_params(seed):
    flat = torch.tensor(scenes.mlp_init_params(seed), dtype=torch.float64, device=DEV)
    out, at = [], 0
    for shape in ((128, 269), (128,), (128, 128), (128,), (128, 128), (128,), (6, 128), (6,)):
        size = math.prod(shape)
        out.append(flat[at:at + size].reshape(shape).clone())
        at += size
    return out


def _mlp(ps, x):
    for k in range(3):
        x = torch.nn.functional.gelu(x @ ps[2 * k].T + ps[2 * k + 1], approximate="tanh")
    return x @ ps[6].T + ps[7]


def _exact_train(case, seed):
    xs, ys, norm = _train_rows(case, seed)
    norm = torch.tensor(norm.astype(np.float64), device=DEV)
    xm, xs_, ym, ys_ = norm[:269], norm[269:538], norm[538:544], norm[544:]
    ps = [p.requires_grad_() for p in _mlp_params(seed)]
    m1 = [torch.zeros_like(p) for p in ps]
    m2 = [torch.zeros_like(p) for p in ps]
    loss = None
    for t in range(1, case["steps"] + 1):
        y = _mlp(ps, (xs[t - 1].double() - xm) / xs_)
        loss = (y - (ys[t - 1].double() - ym) / ys_).square().mean()
        grads = torch.autograd.grad(loss, ps)
        with torch.no_grad():
            for p, g, a, b in zip(ps, grads, m1, m2):
                a.mul_(0.9).add_(g, alpha=0.1)
                b.mul_(0.999).add_(g * g, alpha=0.001)
                p -= TRAIN_LR * (a / (1 - 0.9 ** t)) / ((b / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"params": torch.cat([p.detach().reshape(-1) for p in ps]), "loss": loss.detach()}


def _exact_infer(case, seed):
    ticks, anchors, tau = (t.double() for t in _mlp_rows(case["rows"], seed))
    h, c, rho0 = (float(np.float32(SCENE["h"])), math.sqrt(float(np.float32(SCENE["k"]))), float(np.float32(SCENE["rho0"])))
    w, a, b, d = anchors[:, 3:7].unbind(1)
    rot = torch.stack([1 - 2 * (b * b + d * d), 2 * (a * b - w * d), 2 * (a * d + w * b),
                       2 * (a * b + w * d), 1 - 2 * (a * a + d * d), 2 * (b * d - w * a),
                       2 * (a * d - w * b), 2 * (b * d + w * a), 1 - 2 * (a * a + b * b)], 1).reshape(-1, 3, 3)

    def into(u):                              # R^T u, the anchor's body frame
        return torch.einsum("nij,ni->nj", rot, u)

    cells = anchors[:, 13:].reshape(-1, 64, 4)
    vel = torch.einsum("nij,nki->nkj", rot, cells[:, :, 1:] / c)
    x = torch.cat([into((ticks[:, :3] - anchors[:, :3]) / h), (tau * c / h)[:, None],
                   into((ticks[:, 7:10] - anchors[:, 7:10]) / c), into(ticks[:, 7:10] / c),
                   into(ticks[:, 10:13] * h / c),
                   torch.cat([cells[:, :, :1] / rho0 - 1, vel], 2).reshape(-1, 256)], 1)
    return {"x": x, "y": _mlp(_mlp_params(seed), x / 0.5) * float(np.float32(0.02))}
