"""Tiles of more receiver planes than have coverage bits of their own at a time
(8 for a warp, 28 for a block on 64-texel tiles; 1 and 10 on 128-texel tiles),
up to and past the 64 that are drawn in turns, and waves of few tiles, whose
largest go to blocks.  Each must equal the map path bit for bit, and the work
counters must show that no plane was left without bits: a tile that compares
every covered texel with a plane it has no bits for compares most of them."""
import math

import numpy as np
import pytest

from paper_1410_5780_gb300 import pv3d, scenes as S

from parity import run_gpu

pytestmark = pytest.mark.gpu


def _stack(n_mods, n, map_res, tilted):
    """Modules over one another at heights of their own, facing the same way or
    (tilted) each another way, under a canopy of small triangles."""
    rng = np.random.default_rng(n_mods)
    w = S.make_canopy(31, map_res=map_res, n=n, cells=6, n_steps=4)
    cu, cv = 6, 10
    origins, us, vs = [], [], []
    for k in range(n_mods):
        t, az = (rng.uniform(0.0, 0.9), rng.uniform(0.0, 2.0 * math.pi)) if tilted else (0.4, math.pi)
        u = np.array([-math.cos(az), math.sin(az), 0.0])
        down = np.array([math.sin(az), math.cos(az), 0.0])
        us.append(tuple(u))
        vs.append(tuple(-down * math.cos(t) + np.array([0.0, 0.0, 1.0]) * math.sin(t)))
        origins.append((rng.uniform(-1.5, 1.5), rng.uniform(-1.5, 1.5), 0.3 + 2.0 * k / n_mods))
    w.gen = S._gen_from_lists(origins, us, vs, cu, cv, [0] * n_mods, [-1] * n_mods, list(range(n_mods)),
                              [S.standard_layout(cu, cv, 3)], np.zeros((0, 3)))
    return w


@pytest.mark.parametrize("tilted", [False, True])
@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("n_mods", [9, 11, 29, 40, 65, 90])
def test_many_planes(n_mods, tile, tilted):
    w = _stack(n_mods, 3, 128, tilted)
    outputs = ("cell_counts", "sample_bits", "power", "energy")
    with pv3d.Context(device=0, tile=tile) as c:
        gid = pv3d.load_workload(c, w)
        f = run_gpu(c, gid, w, outputs=outputs)
        m = run_gpu(c, gid, w, outputs=outputs, path=pv3d.PV3D_PATH_MAP)
    for k in outputs:
        np.testing.assert_array_equal(f[k], m[k], err_msg=f"{n_mods} planes, tile {tile}: {k}")
    assert 0 < f["cell_counts"].sum() < f["cell_counts"].size * w.n * w.n


@pytest.mark.parametrize("tile", [64, 128])
def test_every_plane_has_bits(tile):
    """36 parallel modules exactly above one another: along a row a triangle is
    in one relation to each plane, so but for rows of a few texels (some 6 of
    80, at a triangle's tips) nothing is compared texel by texel.  A plane
    without bits compares every texel."""
    w = _stack(36, 3, 512, False)
    w.gen.origin[:, :2] = (0.47, 0.8)
    with pv3d.Context(device=0, tile=tile) as c:
        gid = pv3d.load_workload(c, w)
        c.evaluate(gid, n=w.n, map_res=w.map_res, profile=2)
        p = c.last_profile()
    assert p["texel_visits"] > 0
    assert p["texel_writes"] - p["texel_visits"] < 0.1 * p["texel_visits"], p


@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("n", [1, 2, 5])
def test_few_samples_in_large_cells(n, tile):
    """Cells of some 26 x 26 texels: 27 texels a sample for n = 5, where a
    cell's samples are looked up without a look at its box, and up to 680."""
    w = _stack(12, n, 1024, True)
    outputs = ("cell_counts", "sample_bits", "power")
    with pv3d.Context(device=0, tile=tile) as c:
        gid = pv3d.load_workload(c, w)
        f = run_gpu(c, gid, w, outputs=outputs)
        m = run_gpu(c, gid, w, outputs=outputs, path=pv3d.PV3D_PATH_MAP)
    for k in outputs:
        np.testing.assert_array_equal(f[k], m[k], err_msg=f"n {n}, tile {tile}: {k}")
    assert 0 < f["cell_counts"].sum() < f["cell_counts"].size * n * n


@pytest.mark.parametrize("tile", [32, 64, 128])
def test_suns_along_the_plane_shade_some_and_light_some(tile):
    """The steps with the sun within a degree of the modules' plane (no plane to
    compare with), taken by themselves."""
    from test_gpu_coverage import CASES
    w = CASES["grazing"]()
    w.map_res = max(w.map_res, tile)
    normal = np.cross(w.gen.u[0], w.gen.v[0]).astype(np.float64)
    near = np.abs(w.sun.xyz @ normal) < math.sin(math.radians(1.0))
    assert near.sum() >= 5
    with pv3d.Context(device=0, tile=tile) as c:
        gid = pv3d.load_workload(c, w)
        f = run_gpu(c, gid, w, outputs=("cell_counts",))["cell_counts"][near].astype(np.int64)
        m = run_gpu(c, gid, w, outputs=("cell_counts",), path=pv3d.PV3D_PATH_MAP)["cell_counts"][near]
    np.testing.assert_array_equal(f, m)
    assert 0 < f.sum() < f.size * w.n * w.n
