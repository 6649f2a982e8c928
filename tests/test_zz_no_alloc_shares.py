"""pv3d_module_shade_noalloc where many triangles are just large enough for the
list of large ones: their cost follows their texels, and which of the two
kernels draws a triangle changes no count."""
import numpy as np
import pytest

from paper_1410_5780_gb300 import pv3d

pytestmark = pytest.mark.gpu


def _call(tri, map_res, reps=1):
    """Counts, and the shortest time of a call in milliseconds, of a horizontal
    module of 6 x 10 cells under a zenith sun."""
    import torch
    t = torch.tensor(np.ascontiguousarray(tri, np.float32).reshape(-1, 9), device="cuda:0")
    counts = torch.empty(60, dtype=torch.int32, device="cuda:0")
    module = dict(origin=(0.0, 0.0, 0.0), u=(1.0, 0.0, 0.0), v=(0.0, 1.0, 0.0), pitch=0.15, cells_u=6, cells_v=10)
    best = float("inf")
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        assert pv3d.pv3d_module_shade_noalloc(t, module, np.array([0.0, 0.0, 1.0]), 4, map_res, counts,
                                              torch.cuda.current_stream().cuda_stream) == pv3d.PV3D_OK
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return counts.cpu().numpy(), best


def _scattered(rng, k, texels, map_res):
    """k triangles of `texels` (one number or one each) in width and height
    above the module."""
    side = np.broadcast_to(np.asarray(texels, np.float64) * 1.5 / (map_res - 2), (k,))[:, None, None]
    centre = np.stack([rng.uniform(0.1, 0.8, k), rng.uniform(0.1, 1.4, k), rng.uniform(1.0, 3.0, k)], 1)
    shape = np.array([[-0.5, -0.5, 0.0], [0.5, -0.5, 0.0], [0.0, 0.5, 0.0]])
    return centre[:, None, :] + side * shape + rng.uniform(-0.02, 0.02, (k, 3, 1)) * np.array([0.0, 0.0, 1.0])


def test_cost_follows_the_texels():
    pv3d.load(build_if_missing=True)
    rng = np.random.default_rng(1)
    below = _call(_scattered(rng, 4096, 29, 2048), 2048, reps=12)[1]
    above = _call(_scattered(rng, 4096, 36, 2048), 2048, reps=12)[1]
    # 1.5 times the texels; a warp for every row of the map was 35 times the time
    assert above < 5.0 * below


@pytest.mark.parametrize("map_res", [128, 2048])
def test_order_changes_no_count(map_res):
    """7,000 triangles of one to hundreds of texels, more of them listed than
    the list holds: another order lists others."""
    pv3d.load(build_if_missing=True)
    rng = np.random.default_rng(2)
    tri = _scattered(rng, 7000, np.exp(rng.uniform(np.log(8.0), np.log(90.0), 7000)), map_res)
    tri[:200] = _scattered(rng, 200, np.exp(rng.uniform(0.0, np.log(map_res), 200)), map_res)
    keep = tri[rng.permutation(7000)[:900]]  # fewer than the list holds
    one = _call(keep, map_res)[0]
    assert one.sum() > 0
    np.testing.assert_array_equal(_call(keep[::-1], map_res)[0], one)
    np.testing.assert_array_equal(_call(np.concatenate([np.tile(keep[:100], (50, 1, 1)), keep]), map_res)[0], one)
    np.testing.assert_array_equal(_call(tri[rng.permutation(7000)], map_res)[0], _call(tri, map_res)[0])
