"""GPU parity of the fused path's coverage bits at the sizes where they can go
wrong: tiles of more receiver planes than have bits of their own, suns within
a degree of a module's plane (no plane to compare with: every texel is left
open), modules seen from behind, occluders that cross or touch a receiver's
plane, cells of more than 8 texels and of less than one, and the tile record
pool's overflow.  Each case must equal the map path (depth map + texel
gathers) bit for bit, and the counts must hold shaded samples."""
import math

import numpy as np
import pytest

from paper_1410_5780_gb300 import pv3d, scenes as S

from parity import run_gpu

pytestmark = pytest.mark.gpu


def _rows(n_mods, cells, seed, n, map_res, spread=6.0, suns=None, tilt=None, scene=None):
    """``n_mods`` modules of random orientations (a plane each) among boxes and
    poles that cut through them."""
    rng = np.random.default_rng(seed)
    cu, cv = cells
    lay = S.standard_layout(cu, cv, 1)
    origins, us, vs = [], [], []
    for _ in range(n_mods):
        t = rng.uniform(0.0, 1.2) if tilt is None else tilt
        az = rng.uniform(0, 2 * math.pi) if tilt is None else math.pi
        u = np.array([-math.cos(az), math.sin(az), 0.0])
        down = np.array([math.sin(az), math.cos(az), 0.0])
        us.append(tuple(u))
        vs.append(tuple(-down * math.cos(t) + np.array([0, 0, 1.0]) * math.sin(t)))
        origins.append((rng.uniform(-spread, spread), rng.uniform(-spread, spread), rng.uniform(0.5, 4.0)))
    gen = S._gen_from_lists(origins, us, vs, cu, cv, [0] * n_mods, [-1] * n_mods, list(range(n_mods)), [lay],
                            np.zeros((0, 3)))
    if scene is None:
        mb = S.MeshBuilder()
        for _ in range(12):
            c = rng.uniform(-spread, spread, 2)
            d = rng.uniform(0.2, 2.0, 3)
            mb.box((c[0], c[1], 0.0), (c[0] + d[0], c[1] + d[1], 3.0 * d[2]), edge=rng.choice([None, 0.7]))
        for _ in range(6):  # poles through the modules
            o = np.array(origins[int(rng.integers(n_mods))])
            mb.beam(o + [0.3, 0.2, -1.5], o + [0.4, 0.5, 1.5], 0.05)
        scene = mb.build()
    if suns is None:
        suns = []
        while len(suns) < 9:
            s = S.sun_vectors(40.0, np.array([rng.integers(1, 366)]), np.array([rng.uniform(5.0, 19.0)]))[0]
            if s[2] > 0.02:
                suns.append(s)
    xyz = np.array(suns, np.float64)
    xyz /= np.linalg.norm(xyz, axis=1, keepdims=True)
    k = len(xyz)
    sun = S.Sun(xyz=xyz, dni=np.full(k, 800.0, np.float32), dhi=np.full(k, 100.0, np.float32),
                dt_h=np.ones(k, np.float32))
    return S.Workload("rows", scene, gen, sun, None, n, map_res)


def _grazing_suns(tilt, degrees):
    """Suns at the given angles above the plane of south-facing modules."""
    return [(0.6 * math.cos(a), math.sin(tilt - a) * 0.8, max(0.05, abs(math.sin(a)) * 0.2 + 0.3))
            for a in np.radians(degrees)] + [
        # in the plane through east and the module's slope, turned out of it
        tuple(math.cos(a) * np.array([0.8, 0.6 * math.cos(tilt), 0.6 * math.sin(tilt)])
              + math.sin(a) * np.array([0.0, -math.sin(tilt), math.cos(tilt)])) for a in np.radians(degrees)]


CASES = {
    # more planes in a tile than levels (12, 8 and 4): the last level is shared
    "planes_32": lambda: _rows(40, (4, 5), 3, 4, 64),
    "planes_32_fine": lambda: _rows(24, (6, 10), 4, 3, 512),
    # the sun within a degree of the modules' plane, on it, and behind it
    "grazing": lambda: _rows(6, (6, 10), 5, 4, 256, spread=2.0, tilt=0.5,
                             suns=_grazing_suns(0.5, [-40.0, -2.0, -0.9, -0.1, 0.0, 0.1, 0.9, 1.1, 5.0])),
    # cells of many texels (their rows span words and tiles), and of less than one
    "big_cells": lambda: _rows(2, (3, 2), 6, 8, 1024, spread=0.6),
    "big_cells_n15": lambda: _rows(2, (2, 3), 7, 15, 512, spread=0.6),
    "small_cells": lambda: _rows(9, (6, 12), 8, 5, 64, spread=8.0),
    # many small triangles across one plane: more open triangles than a warp lists
    "canopy": lambda: S.make_canopy(31, map_res=128, cells=40),
}


@pytest.mark.parametrize("u24", [False, True])
@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("case", sorted(CASES))
def test_coverage_equals_map(case, tile, u24):
    w = CASES[case]()
    w.map_res = max(w.map_res, tile)  # (a map smaller than a tile has no tiles)
    fmt = pv3d.PV3D_DEPTH_U24 if u24 else pv3d.PV3D_DEPTH_F32
    outputs = ("cell_counts", "power", "energy", "cell_beam_loss") + (("sample_bits",) if w.n <= 8 else ())
    with pv3d.Context(device=0, tile=tile, depth_format=fmt) as c:
        gid = pv3d.load_workload(c, w)
        f = run_gpu(c, gid, w, outputs=outputs)
        m = run_gpu(c, gid, w, outputs=outputs, path=pv3d.PV3D_PATH_MAP)
        # without a per-cell output only the cells near covered texels are looked at
        e = run_gpu(c, gid, w, outputs=("power", "energy"))
    for k in outputs:
        np.testing.assert_array_equal(f[k], m[k], err_msg=f"{case} {tile}: {k}")
    for k in ("power", "energy"):
        np.testing.assert_array_equal(e[k], f[k], err_msg=f"{case} {tile}: {k} without per-cell outputs")
    assert f["cell_counts"].sum() > 0
    if case == "grazing":
        assert (f["cell_counts"] < w.n * w.n).any()


def test_crossing_planes_equal_map():
    """Plates that cut through a module at its own depth, tilted a little
    against it: the band where depths are compared runs along the module."""
    tilt = 0.4
    mb = S.MeshBuilder()
    up = np.array([0.0, math.cos(tilt), math.sin(tilt)])
    normal = np.array([0.0, -math.sin(tilt), math.cos(tilt)])
    for k, eps in enumerate((1e-4, 1e-3, 1e-2, 0.1)):
        p0 = np.array([0.1 + 0.25 * k, 0.0, 1.0]) + 0.2 * up - eps * normal
        mb.grid_quad(p0, (0.2, 0.0, 0.0), 1.2 * up + 2 * eps * normal, 1, 3)
    w = _rows(1, (8, 10), 9, 6, 512, spread=0.0, tilt=tilt, scene=mb.build())
    w.gen.origin[:] = (0.0, 0.0, 1.0)
    for tile in (32, 64, 128):
        with pv3d.Context(device=0, tile=tile) as c:
            gid = pv3d.load_workload(c, w)
            f = run_gpu(c, gid, w, outputs=("cell_counts", "sample_bits", "power"))
            m = run_gpu(c, gid, w, outputs=("cell_counts", "sample_bits", "power"), path=pv3d.PV3D_PATH_MAP)
        for k in ("cell_counts", "sample_bits", "power"):
            np.testing.assert_array_equal(f[k], m[k], err_msg=f"tile {tile}: {k}")
        assert 0 < (f["sample_bits"] != 0).sum()
