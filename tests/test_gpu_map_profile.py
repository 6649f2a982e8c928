"""Work counters of the map path (profile bit 1)."""
import numpy as np
import pytest

from paper_1410_5780_gb300 import pv3d, scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,map_res,dense", [(15, 64, True), (2, 1024, False)])
def test_map_path_counts_its_work(n, map_res, dense):
    """Samples far more than texels: tiles drawn at every texel, nothing marked.
    Far fewer: every sample of a tile looked at to mark its texel."""
    w = S.make_canopy(31, map_res=map_res, n=n, cells=20)
    with pv3d.Context(device=0, tile=64) as c:
        gid = pv3d.load_workload(c, w)
        r = c.evaluate(gid, n=n, map_res=map_res, outputs=("cell_counts",), path=pv3d.PV3D_PATH_MAP, profile=2)
        p = c.last_profile()
    shaded = int(np.asarray(r["cell_counts"].cpu()).sum())
    assert 0 < shaded <= p["sample_tests"] <= r["tests"]
    if dense:
        assert 0 < p["dense_tiles"] <= p["nonempty_tiles"]
    else:
        assert p["dense_tiles"] == 0
        assert p["candidates"] >= p["sample_tests"]
