"""Binning by boxes of boxes: meshlets in groups of 32 tested against the light
window together, and meshlets over many tiles tested against blocks of tiles.
Triangles far beside the light window must change nothing, however many groups
of meshlets they fill, and neither must the tile size, which decides how many
tiles a meshlet covers (R = 2048: 4096 tiles of 32 texels, 256 of 128)."""
import numpy as np
import pytest

from paper_1410_5780_gb300 import pv3d, scenes as S

from parity import run_gpu
from test_gpu_coverage import _rows

pytestmark = pytest.mark.gpu

OUT = ("cell_counts", "sample_bits", "power", "energy")


def _scene(extra, roof):
    """Boxes beside the modules, `extra` triangles half a kilometre east below
    the horizon, and a roof over the field in one grid of roof x roof quads with
    gaps (its meshlets span the window)."""
    mb = S.MeshBuilder()
    rng = np.random.default_rng(5)
    for _ in range(10):
        c, d = rng.uniform(-6, 6, 2), rng.uniform(0.3, 2.0, 3)
        mb.box((c[0], c[1], 0.0), (c[0] + d[0], c[1] + d[1], 3.0 * d[2]))
    for k in range(roof):
        mb.grid_quad((-7.0, -7.0 + 14.0 * k / roof, 6.0), (14.0, 0.0, 0.3), (0.0, 3.0 / roof, 0.0), 2, 1)
    if extra:
        mb.grid_quad((500.0, -40.0, -20.0), (60.0, 0.0, 0.0), (0.0, 80.0, 0.0), 1, (extra + 1) // 2)
    return mb.build()


def _run(scene, tile, map_res, path=0):
    w = _rows(12, (4, 5), 11, 4, map_res, scene=scene)
    with pv3d.Context(device=0, tile=tile) as c:
        gid = pv3d.load_workload(c, w)
        return run_gpu(c, gid, w, outputs=OUT, path=path)


@pytest.mark.parametrize("extra", [800, 1024, 3400, 70000])
def test_far_groups_change_nothing(extra):
    base, more = (_run(_scene(e, 3), 32, 512) for e in (0, extra))
    assert base["cell_counts"].sum() > 0
    for k in OUT:
        np.testing.assert_array_equal(more[k], base[k], err_msg=k)


@pytest.mark.parametrize("path", [pv3d.PV3D_PATH_FUSED, pv3d.PV3D_PATH_MAP])
def test_tile_blocks_change_nothing(path):
    scene = _scene(3000, 24)
    want = _run(scene, 128, 2048, path)
    assert want["cell_counts"].sum() > 0
    for tile in (32, 64):
        got = _run(scene, tile, 2048, path)
        for k in OUT:
            np.testing.assert_array_equal(got[k], want[k], err_msg=f"{tile} {k}")
