"""Workloads of the shadow-sample library, for timing it and for comparing two
builds of it: what a user has it compute, through the public binding
(paper_1410_5780_gb300.pv3d).

``listed()`` names them, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes the inputs and the context a user's program keeps, ``run`` is
one call on them, ``work`` what that call cannot do without and ``exact`` the
values plain numpy gives in 64 bits.  Scenes, generators and sun tables come
from the seeded builders of paper_1410_5780_gb300.scenes; every seed gives
another scene.

A case's shadow-map side, samples per cell side, tile side and steps per wave
are the user's choices: the tuned ones of the benchmark for the large plants
(tile 32 or 128, 256 steps), the library's defaults elsewhere (0).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1410_5780_gb300 import pv3d, scenes

I_REF, V_CELL, V_DIODE = 9.0, 0.5, 0.5  # the library's defaults: A at 1000 W/m^2, V, V
ENERGY = ("energy", "energy_unshaded")
POWER = ENERGY + ("power", "power_unshaded")
COUNTS = POWER + ("cell_counts",)
REPORT = ENERGY + ("cell_beam_loss", "string_energy", "string_energy_unshaded", "array_energy",
                   "array_energy_unshaded")


def listed():
    return [
        # One module, one sun, no allocation: the call a latency-critical loop
        # makes, with the few thousand triangles around a house.
        dict(name="module_now", kind="module", tris=2000, cells_u=6, cells_v=10, n=4, map_res=512),
        # The smallest evaluation: two modules before a box over the 24 hours of
        # a day, as an interactive planner asks for it after each change.
        dict(name="day_plan", kind="tiny", n=4, map_res=1024),
        # A few tracked modules among boxes and poles: odd counts, 5 x 5 samples,
        # 24-bit depth, every per-step output and the sample flags.
        dict(name="rows_odd", kind="rows", modules=13, boxes=9, cells_v=12, steps=45, n=5, map_res=512, tracked=True,
             u24=True),
        # The building-integrated facade over an hourly year (the benchmark's
        # second workload): module energies and the power of every hour.
        dict(name="facade_year", kind="facade", floors=8, per_floor=25, tris=50000, day=1, days=365, step_h=1.0, n=8,
             map_res=4096, tile=128, chunk=256, report=False, u24=False),
        # The same year as a yield report: strings of five modules, five strings
        # an inverter input, the loss of every cell and the sky map of the
        # losses, with the library's default tile and wave.
        dict(name="facade_report", kind="facade", floors=8, per_floor=25, tris=50000, day=1, days=365, step_h=1.0, n=8,
             map_res=4096, tile=0, chunk=0, report=True, u24=False),
        # The tracker plant over a quarter-hour year: the benchmark's headline.
        dict(name="tracker_year", kind="tracker", gx=25, gy=20, terrain=512, pylons=20, day=1, days=365, step_h=0.25,
             n=4, map_res=8192, tile=32, chunk=256, windows=False, u24=False, counts=False),
        # One spring day of that plant, with the shaded samples of every cell.
        dict(name="tracker_day", kind="tracker", gx=25, gy=20, terrain=512, pylons=20, day=80, days=1, step_h=0.25,
             n=4, map_res=8192, tile=32, chunk=256, windows=False, u24=True, counts=True),
        # A light window of its own for each tracker (finer texels).
        dict(name="tracker_windows", kind="tracker", gx=25, gy=20, terrain=512, pylons=20, day=172, days=1, step_h=0.5,
             n=4, map_res=256, tile=32, chunk=256, windows=True, u24=False, counts=False),
        # The diffuse term: the sky seen by every cell of the facade, then a
        # month with that shading.
        dict(name="diffuse_month", kind="sky", floors=8, per_floor=25, tris=50000, day=152, days=30, step_h=1.0, n=8,
             map_res=4096, rings=9, sectors=36),
        # Many sites of uneven size in one call (a portfolio).
        dict(name="batch_mix", kind="batch", scenes=16, tris_lo=1000, tris_hi=200000, mods_lo=10, mods_hi=2000,
             steps_lo=100, steps_hi=4400, n=4, u24=False),
        # A plant from host arrays to host results in one go: scene, generator,
        # sun and poses loaded, two days evaluated, everything released.
        dict(name="project", kind="project", gx=25, gy=20, terrain=512, pylons=20, day=300, days=2, step_h=0.25, n=4,
             map_res=8192, tile=32, chunk=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2(x, lo, hi):
    r = lo
    while r < x and r < hi:
        r *= 2
    return r


def draw(rng):
    kind = rng.choice(("module", "rows", "facade", "facade", "tracker", "tracker", "sky", "batch", "project"))
    if kind == "module":
        return dict(kind=kind, tris=_log_int(rng, 12, 20000), cells_u=rng.randint(3, 12), cells_v=rng.randint(4, 16),
                    n=rng.randint(2, 9), map_res=rng.choice((256, 512, 1024, 2048)))
    if kind == "rows":
        return dict(kind=kind, modules=_log_int(rng, 3, 60), boxes=rng.randint(3, 25),
                    cells_v=rng.choice((8, 10, 12)), steps=_log_int(rng, 5, 400), n=rng.randint(2, 8), map_res=rng.choice((512, 1024, 2048)), tracked=rng.random() < 0.5,
                    u24=rng.random() < 0.3)
    if kind in ("facade", "sky"):
        c = dict(kind=kind, floors=rng.randint(2, 12), per_floor=rng.randint(5, 40), tris=_log_int(rng, 4000, 120000),
                 day=rng.randint(1, 300), days=_log_int(rng, 1, 64), step_h=rng.choice((0.25, 0.5, 1.0)),
                 n=rng.randint(2, 8), map_res=rng.choice((1024, 2048, 4096)))
        if kind == "sky":
            return dict(c, rings=rng.randint(5, 12), sectors=rng.randint(11, 40))
        return dict(c, tile=rng.choice((0, 32, 128)), chunk=rng.choice((0, 100, 256)), report=rng.random() < 0.4,
                    u24=rng.random() < 0.3)
    if kind in ("tracker", "project"):
        gx, gy = rng.randint(3, 25), rng.randint(3, 20)
        windows = kind == "tracker" and rng.random() < 0.25
        c = dict(kind=kind, gx=gx, gy=gy, terrain=_log_int(rng, 64, 512), pylons=rng.randint(0, 12),
                 day=rng.randint(1, 360), days=rng.randint(1, 4), step_h=rng.choice((0.25, 0.5, 1.0)),
                 n=rng.randint(2, 6), map_res=256 if windows else _pow2(max(gx, gy) * 24 / 0.075, 1024, 8192),
                 tile=rng.choice((0, 32)), chunk=rng.choice((0, 200, 256)))
        if kind == "project":
            return c
        return dict(c, windows=windows, u24=rng.random() < 0.3, counts=not windows and rng.random() < 0.5)
    return dict(kind=kind, scenes=rng.randint(3, 24), tris_lo=1000, tris_hi=_log_int(rng, 8000, 200000), mods_lo=10,
                mods_hi=_log_int(rng, 40, 1500), steps_lo=50, steps_hi=_log_int(rng, 200, 2000), n=rng.randint(3, 5),
                u24=rng.random() < 0.3)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _workload(c, seed):
    """The scenes.Workload of a case of one generator, under the seed's weather:
    a measured series in place of the clear sky."""
    w = _site(c, seed)
    rng = np.random.default_rng(seed)
    w.sun.dni = (w.sun.dni * rng.uniform(0.2, 1.0, w.sun.n_steps)).astype(np.float32)
    w.sun.dhi = (w.sun.dhi * rng.uniform(0.8, 2.5, w.sun.n_steps)).astype(np.float32)
    return w


def _site(c, seed):
    kind = c["kind"]
    if kind == "tiny":
        w = scenes.make_tiny(day=1 + (37 * seed) % 365, n=c["n"], map_res=c["map_res"])
        w.scene.verts[:, 0] += np.float32(0.01 * (seed % 90))  # the box, moved sideways
        return w
    if kind == "rows":
        for k in range(1000):  # the seed's first scene with the case's module height
            w = scenes.make_random_small([seed, k], n_mods=c["modules"], n_boxes=c["boxes"], n_steps=c["steps"],
                                         n=c["n"], map_res=c["map_res"], tracked=c["tracked"])
            if int(w.gen.cells_v[0]) == c["cells_v"]:
                return w
        raise RuntimeError("no scene with that module height")
    days = np.arange(c["day"], c["day"] + c["days"])
    if kind in ("facade", "sky"):
        w = scenes.make_facade(seed=seed, n=c["n"], map_res=c["map_res"], floors=c["floors"], per_floor=c["per_floor"],
                               target_tris=c["tris"], step_h=c["step_h"], days=days)
        w.gen.string = (np.arange(w.gen.n_modules) // 5).astype(np.int32)
        w.gen.array = (np.arange(w.gen.n_modules) // 25).astype(np.int32)
        return w
    # tracker plants: 24 m between trackers, as on the 25 x 20 plant
    spacing = (24.0 * max(c["gx"], c["gy"]) + 13.2) / (c["terrain"] - 1)
    return scenes.make_tracker(seed=seed, n=c["n"], map_res=c["map_res"], grid=(c["gx"], c["gy"]),
                               terrain_n=c["terrain"], spacing=spacing, n_pylons=c["pylons"], step_h=c["step_h"],
                               days=days)


def _module_inputs(c, seed):
    """Triangles scattered around one tilted module (a third of them in the
    sun's way), the module and a daytime sun."""
    rng = np.random.default_rng(seed)
    tilt, el, az = np.radians([rng.uniform(10, 40), rng.uniform(20, 70), rng.uniform(120, 240)])
    sun = np.array([math.cos(el) * math.sin(az), math.cos(el) * math.cos(az), math.sin(el)])
    sun /= np.linalg.norm(sun)
    pitch = scenes.CELL_PITCH
    module = dict(origin=(0.0, 0.0, 0.5), u=(1.0, 0.0, 0.0), v=(0.0, math.cos(tilt), math.sin(tilt)), pitch=pitch,
                  cells_u=c["cells_u"], cells_v=c["cells_v"])
    t = c["tris"]
    centre = rng.uniform(-12.0, 12.0, (t, 3))
    k = t // 3
    mid = np.array([0.5 * pitch * c["cells_u"], 0.4 * pitch * c["cells_v"], 0.8])
    centre[:k] = mid + sun * rng.uniform(1.0, 12.0, (k, 1)) + rng.normal(0.0, 0.8, (k, 3))
    centre[:, 2] = np.abs(centre[:, 2]) + 0.2
    tri = centre[:, None, :] + rng.normal(0.0, 0.15, (t, 3, 3))
    return module, sun, tri.astype(np.float32)


def _batch(c, seed):
    """Facade-like and tracker-like sites in turn: the case fixes how many
    triangles, modules and steps each has (log-uniform, steps uniform), the
    seed what stands there and where on Earth."""
    sizes = np.random.default_rng(4)
    out = []
    for q in range(c["scenes"]):
        tris = int(math.exp(sizes.uniform(math.log(c["tris_lo"]), math.log(c["tris_hi"]))))
        mods = int(math.exp(sizes.uniform(math.log(c["mods_lo"]), math.log(c["mods_hi"]))))
        steps = int(sizes.integers(c["steps_lo"], c["steps_hi"] + 1))
        for k in range(64):  # the builder tosses a coin for the kind of site
            rng = np.random.default_rng([seed, q, k])
            w = scenes.make_mixed_scene(rng, tris, mods, float(rng.uniform(0.0, 60.0)), steps, n=c["n"])
            if (w.gen.pivots.shape[0] > 0) == (q % 2 == 1):
                break
        out.append(w)
    return out


def _outputs(c):
    kind = c["kind"]
    if kind == "rows":
        return COUNTS + ("sample_bits",)
    if kind == "tiny":
        return COUNTS
    if kind == "facade":
        return REPORT if c["report"] else POWER
    if kind == "tracker":
        return ENERGY + ("cell_counts",) if c["counts"] else ENERGY
    return ENERGY


def _context(c):
    return pv3d.Context(tile=c.get("tile", 0), chunk_steps=c.get("chunk", 0),
                        depth_format=pv3d.PV3D_DEPTH_U24 if c.get("u24") else pv3d.PV3D_DEPTH_F32)


def prepare(case, seed):
    c = case
    if c["kind"] == "module":
        module, sun, tri = _module_inputs(c, seed)
        return dict(case=c, module=module, sun=sun, tri=torch.from_numpy(tri.reshape(-1)).cuda(),
                    counts=torch.zeros(c["cells_u"] * c["cells_v"], dtype=torch.int32, device="cuda"))
    ctx = _context(c)
    if c["kind"] == "batch":
        ws = _batch(c, seed)
        return dict(case=c, ctx=ctx, gens=[pv3d.load_workload(ctx, w) for w in ws], map_res=[w.map_res for w in ws])
    w = _workload(c, seed)
    if c["kind"] == "project":
        return dict(case=c, ctx=ctx, workload=w)
    return dict(case=c, ctx=ctx, gen=pv3d.load_workload(ctx, w))


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "module":
        rc = pv3d.pv3d_module_shade_noalloc(state["tri"], state["module"], state["sun"], c["n"], c["map_res"],
                                            state["counts"], torch.cuda.current_stream().cuda_stream)
        if rc != pv3d.PV3D_OK:
            raise RuntimeError(f"pv3d_module_shade_noalloc: {rc}")
        return dict(counts=state["counts"])
    ctx = state["ctx"]
    if kind == "batch":
        got = ctx.evaluate_batch(state["gens"], n=c["n"], map_res=state["map_res"])
        return [{k: r[k] for k in ENERGY} for r in got]
    if kind == "project":
        w = state["workload"]
        scene = ctx.scene_load(w.scene.verts, w.scene.tris)
        gen = ctx.generator_define(scene, w.gen)
        ctx.set_sun(gen, w.sun.xyz, w.sun.dni, w.sun.dhi, w.sun.dt_h)
        ctx.set_poses(gen, w.poses)
        r = ctx.evaluate(gen, n=c["n"], map_res=c["map_res"], outputs=ENERGY, device=False)
        ctx.release(gen)
        ctx.release(scene)
        return {k: r[k] for k in ENERGY}
    gen = state["gen"]
    if kind == "sky":
        f = ctx.sky_view(gen, rings=c["rings"], sectors=c["sectors"], n=c["n"], map_res=c["map_res"])
        r = ctx.evaluate(gen, n=c["n"], map_res=c["map_res"], outputs=POWER, diffuse_shading=True)
        return dict({k: r[k] for k in POWER}, fraction=f)
    outputs = _outputs(c)
    heat = (36, 9) if c.get("report") else None
    r = ctx.evaluate(gen, n=c["n"], map_res=c["map_res"], outputs=outputs, heat_bins=heat,
                     window_groups=pv3d.PV3D_WINDOWS_PER_TRACKER if c.get("windows") else pv3d.PV3D_WINDOWS_ONE)
    if heat:
        outputs = outputs + ("heat_energy", "heat_energy_unshaded", "heat_steps")
    return {k: r[k] for k in outputs}


# ---------------------------------------------------------------------------
# what a call cannot do without
# ---------------------------------------------------------------------------
TEST_FLOPS = 14  # of one sample test: its position, projection and texel, and the compare


def _work_of(w, outputs, steps, heat=False):
    g = w.gen
    m, cells, lit = g.n_modules, g.n_cells, int((w.sun.xyz[:, 2] > 0).sum())
    strings, arrays = len(np.unique(g.string)), 1 if g.array is None else len(np.unique(g.array))
    size = dict(energy=8 * m, energy_unshaded=8 * m, power=4 * steps * m, power_unshaded=4 * steps * m,
                cell_counts=steps * cells, sample_bits=8 * steps * cells, cell_beam_loss=8 * cells,
                string_energy=8 * strings, string_energy_unshaded=8 * strings, array_energy=8 * arrays,
                array_energy_unshaded=8 * arrays)
    read = 36 * w.scene.n_tris + 64 * m + 36 * steps + 8 * steps * g.pivots.shape[0]
    return dict(bytes=read + sum(size[k] for k in outputs) + (36 * 9 * 20 if heat else 0),
                flops=TEST_FLOPS * lit * w.samples_per_step)


def work(case):
    c = case
    if c["kind"] == "module":
        cells = c["cells_u"] * c["cells_v"]
        return dict(bytes=36 * c["tris"] + 4 * cells, flops=30 * c["tris"] + TEST_FLOPS * cells * c["n"] ** 2)
    if c["kind"] == "batch":
        each = [_work_of(w, ENERGY, w.sun.n_steps) for w in _batch(c, 0)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    w = _workload(c, 0)
    if c["kind"] == "sky":
        d = _work_of(w, POWER, w.sun.n_steps)
        patches = c["rings"] * c["sectors"]
        return dict(bytes=d["bytes"] + 4 * w.gen.n_cells,
                    flops=d["flops"] + TEST_FLOPS * patches * w.samples_per_step)
    return _work_of(w, _outputs(c), w.sun.n_steps, heat=bool(c.get("report")))


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def _normals(w):
    n = np.cross(w.gen.u.astype(np.float64), w.gen.v.astype(np.float64))
    return n / np.linalg.norm(n, axis=1, keepdims=True)


def _rotation(az, tilt):
    """Rz(pi - az) Rx(tilt), [..., 3, 3]."""
    cg, sg, cb, sb = -np.cos(az), np.sin(az), np.cos(tilt), np.sin(tilt)
    z = np.zeros_like(cg)
    return np.stack([np.stack([cg, -sg * cb, sg * sb], -1), np.stack([sg, cg * cb, -cg * sb], -1),
                     np.stack([z, sb, cb], -1)], -2)


def _irradiance(w):
    """Beam and diffuse irradiance of each orientation, [steps, orientations],
    and the orientation of each module (a tracker's modules that face one way,
    the fixed modules that do)."""
    g, s = w.gen, w.sun
    lit = s.xyz[:, 2] > 0
    faces, of_module = np.unique(np.column_stack([g.tracker, _normals(w)]), axis=0, return_inverse=True)
    cosi, nz = np.empty((s.n_steps, len(faces))), np.empty((s.n_steps, len(faces)))
    for q, face in enumerate(faces):
        normal = face[1:]
        if face[0] >= 0:
            pose = w.poses[:, int(face[0])].astype(np.float64)
            normal = _rotation(pose[:, 0], pose[:, 1]) @ normal
        cosi[:, q] = (s.xyz * normal).sum(1)
        nz[:, q] = normal[..., 2]
    dni = np.where(lit, s.dni.astype(np.float64), 0.0)[:, None]
    dhi = np.where(lit, s.dhi.astype(np.float64), 0.0)[:, None]
    return dni * np.maximum(cosi, 0.0), dhi * (1.0 + nz) * 0.5, of_module.reshape(-1)


def _shaded_counts(w):
    """Shaded samples per cell, [steps, cells], by a ray toward the sun from
    every sample against every triangle and module: the surface itself, where
    the library takes its depth from a map."""
    g, s, n = w.gen, w.sun, w.n
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    u, v = g.u.astype(np.float64), g.v.astype(np.float64)
    tri = w.scene.verts.astype(np.float64)[w.scene.tris]
    counts = np.zeros((s.n_steps, g.n_cells))
    for k in range(s.n_steps):
        sun = s.xyz[k]
        if not sun[2] > 0:
            continue
        quads, samples = [], []
        for m in range(g.n_modules):
            o, du, dv = g.origin[m].astype(np.float64), u[m], v[m]
            t = int(g.tracker[m])
            if t >= 0:
                rot = _rotation(*w.poses[k, t].astype(np.float64))
                o, du, dv = g.pivots[t].astype(np.float64) + rot @ o, rot @ du, rot @ dv
            p, cu, cv = float(g.pitch[m]), int(g.cells_u[m]), int(g.cells_v[m])
            quads.append((o, du * (cu * p), dv * (cv * p)))
            a, b = (np.arange(cu * n) + 0.5) * p / n, (np.arange(cv * n) + 0.5) * p / n
            samples.append(o + a[None, :, None] * du + b[:, None, None] * dv)
        cell = 0
        for m in range(g.n_modules):
            own = [np.stack([o, o + a, o + a + b]) for q, (o, a, b) in enumerate(quads) if q != m]
            own += [np.stack([o, o + a + b, o + b]) for q, (o, a, b) in enumerate(quads) if q != m]
            rays = torch.from_numpy(samples[m].reshape(-1, 3)).to(dev)
            hit = torch.zeros(rays.shape[0], dtype=torch.bool, device=dev)
            every = torch.from_numpy(np.concatenate([tri, np.stack(own)]) if own else tri).to(dev)
            e1, e2 = every[:, 1] - every[:, 0], every[:, 2] - every[:, 0]
            d = torch.from_numpy(sun).to(dev)
            h = torch.linalg.cross(d.expand_as(e2), e2)
            det = (e1 * h).sum(1)
            ok = det.abs() > 1e-14
            inv = torch.where(ok, 1.0 / torch.where(ok, det, torch.ones_like(det)), torch.zeros_like(det))
            for r0 in range(0, rays.shape[0], 4096):
                q = rays[r0:r0 + 4096, None, :] - every[None, :, 0]
                x = (q * h).sum(2) * inv
                c = torch.linalg.cross(q, e1[None].expand_as(q))
                y = (c @ d) * inv
                t = (c * e2).sum(2) * inv
                hit[r0:r0 + 4096] = (ok & (x >= 0) & (y >= 0) & (x + y <= 1) & (t > 1e-4)).any(1)
            cu, cv = int(g.cells_u[m]), int(g.cells_v[m])
            per = hit.cpu().numpy().reshape(cv, n, cu, n).sum((1, 3)).reshape(-1)
            counts[k, cell:cell + cu * cv] = per
            cell += cu * cv
    return counts


def _shaded_power(w, counts):
    """Module power at the best of its bypass states, [steps, modules]."""
    g = w.gen
    beam, diff, face = _irradiance(w)
    power = np.zeros((w.sun.n_steps, g.n_modules))
    cell = 0
    for m in range(g.n_modules):
        nc = int(g.cells_u[m] * g.cells_v[m])
        lay = g.layouts[int(g.layout[m])]
        amps = I_REF * 1e-3 * (beam[:, face[m], None] * (1.0 - counts[:, cell:cell + nc] / w.n ** 2)
                               + diff[:, face[m], None])
        sub = np.stack([amps[:, lay.cell_sub == q].min(1) for q in range(lay.n_sub)], 1)
        cells = np.bincount(lay.cell_sub, minlength=lay.n_sub) * V_CELL
        for q in range(lay.n_sub):
            volt = np.where(sub >= sub[:, q, None], cells, -V_DIODE).sum(1)
            power[:, m] = np.maximum(power[:, m], sub[:, q] * volt)
        cell += nc
    return power


def _exact_of(w, outputs):
    dt = w.sun.dt_h.astype(np.float64)[:, None]
    beam, diff, face = _irradiance(w)
    watts = (w.gen.cells_u * w.gen.cells_v) * (I_REF * V_CELL * 1e-3)  # of a module at 1 W/m^2, unshaded
    got = dict.fromkeys(outputs)
    got["energy_unshaded"] = ((beam + diff) * dt).sum(0)[face] * watts
    if "power_unshaded" in got:
        got["power_unshaded"] = (beam + diff)[:, face] * watts
    pairs = w.samples_per_step * (w.scene.n_tris + 2 * w.gen.n_modules) * w.sun.n_steps
    if "power" in got and pairs <= 2e9:  # samples against triangles: seconds
        p = _shaded_power(w, _shaded_counts(w))
        got["power"] = p
        got["energy"] = (p * dt).sum(0)
    # modules of a string or array of the facade share one plane: without
    # shading one current runs through all of them
    if "string_energy_unshaded" in got:
        got["string_energy_unshaded"] = np.bincount(w.gen.string, weights=got["energy_unshaded"])
    if "array_energy_unshaded" in got and w.gen.n_modules % 5 == 0:  # strings of one length
        got["array_energy_unshaded"] = np.bincount(w.gen.array, weights=got["energy_unshaded"])
    return got


def exact(case, seed):
    c = case
    if c["kind"] == "module":
        return None  # counts: whole numbers
    if c["kind"] == "batch":
        return [_exact_of(w, ENERGY) for w in _batch(c, seed)]
    w = _workload(c, seed)
    if c["kind"] == "sky":
        return dict(_exact_of(w, ENERGY + ("power_unshaded",)), power=None, fraction=None)
    got = _exact_of(w, _outputs(c))
    return dict(got, heat_energy=None, heat_energy_unshaded=None, heat_steps=None) if c.get("report") else got
