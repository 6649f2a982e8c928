"""pv3d_module_shade_noalloc over triangles of all sizes: from one texel to the
whole map (those above 1024 texels go through a list of 4096 to a kernel of
their own, and past its end stay with the first), widths about the powers of
two that share a warp among rows.  Drawing a triangle again changes nothing, so
n copies of it must give the counts of one, whichever way they take."""
import numpy as np
import pytest

from paper_1410_5780_gb300 import pv3d

from test_zz_no_alloc import _one_module_workload

pytestmark = pytest.mark.gpu


def _counts(w, step, tri, map_res):
    import torch
    m = w.gen
    module = dict(origin=m.origin[0], u=m.u[0], v=m.v[0], pitch=float(m.pitch[0]), cells_u=int(m.cells_u[0]),
                  cells_v=int(m.cells_v[0]))
    counts = torch.empty(int(m.cells_u[0] * m.cells_v[0]), dtype=torch.int32, device="cuda:0")
    t = torch.tensor(np.ascontiguousarray(tri, np.float32).reshape(-1, 9), device="cuda:0")
    assert pv3d.pv3d_module_shade_noalloc(t, module, w.sun.xyz[step], w.n, map_res, counts,
                                          torch.cuda.current_stream().cuda_stream) == pv3d.PV3D_OK
    torch.cuda.synchronize()
    return counts.cpu().numpy()


def _triangle(w, step, width, height):
    """A triangle across the light, `width` by `height` of the module's longer
    side, a metre towards the sun from the module's middle."""
    g = w.gen
    s = np.asarray(w.sun.xyz[step], np.float64)
    right = np.array([s[1], -s[0], 0.0]) / np.hypot(s[0], s[1])
    up = np.cross(s, right)
    lu, lv = g.cells_u[0] * g.pitch[0], g.cells_v[0] * g.pitch[0]
    c = g.origin[0] + 0.5 * lu * np.asarray(g.u[0]) + 0.5 * lv * np.asarray(g.v[0]) + s
    e = max(lu, lv)
    return np.array([c - 0.4 * height * e * up, c - 0.4 * height * e * up + width * e * right,
                     c + 0.6 * height * e * up])


@pytest.mark.parametrize("map_res", [64, 512])
@pytest.mark.parametrize("width", [0.02, 0.07, 0.26, 0.5, 3.0])
def test_copies_of_a_triangle(width, map_res):
    pv3d.load(build_if_missing=True)
    w = _one_module_workload()
    step = int(np.argmax(w.sun.xyz[:, 2]))
    for height in (0.1, 1.0, 4.0):
        tri = _triangle(w, step, width, height)
        one = _counts(w, step, tri, map_res)
        for copies in (2, 31, 4200):
            np.testing.assert_array_equal(_counts(w, step, np.tile(tri, (copies, 1, 1)), map_res), one)
    assert one.sum() > 0 or width < 0.1


@pytest.mark.parametrize("width,height", [(0.3, 0.5), (1.0, 1.0), (2.5, 3.0)])
def test_sizes_match_evaluate(width, height):
    import torch
    from paper_1410_5780_gb300 import scenes as S
    w = _one_module_workload()
    step = int(np.argmax(w.sun.xyz[:, 2]))
    tri = _triangle(w, step, width, height)
    mb = S.MeshBuilder()
    mb.add(tri, np.array([[0, 1, 2]]))
    w.scene = mb.build()
    with pv3d.Context(device=0, map_res=512) as ctx:
        gid = pv3d.load_workload(ctx, w)
        r = ctx.evaluate(gid, n=w.n, map_res=512, outputs=("cell_counts",), device=True)
        torch.cuda.synchronize()
        ref = r["cell_counts"].cpu().numpy().astype(np.int64)[step]
    diff = np.abs(_counts(w, step, w.scene.verts[w.scene.tris], 512).astype(np.int64) - ref)
    # a sample whose texel centre lies on an edge may fall either way: one a cell
    assert ref.sum() > 0 and diff.max() <= 1
