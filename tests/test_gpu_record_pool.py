"""The pool of tile records (the coverage bits of the fused path): its first
size stays within the context's memory budget, and a wave that needs more is
run again with a larger pool, evaluated or served, with the same results."""
import numpy as np
import pytest

from paper_1410_5780_gb300 import pv3d, scenes as S

from parity import run_gpu

pytestmark = pytest.mark.gpu

OUTS = ("energy", "power", "cell_counts", "sample_bits")


def _used():
    import torch
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info(0)
    return total - free


def test_first_size_stays_in_the_budget():
    """24 suns over 8192 x 8192 texels: 393,216 tiles, whose records would take
    252 MB if every tile had one."""
    w = S.make_tiny(day=172, n=2, map_res=8192)
    budget = 160 << 20
    with pv3d.Context(device=0, tile=64) as c:  # (the CUDA context and module, before anything is counted)
        run_gpu(c, pv3d.load_workload(c, w), w, outputs=("energy",))
    before = _used()
    with pv3d.Context(device=0, tile=64, hbm_budget_bytes=budget) as c:
        gid = pv3d.load_workload(c, w)
        run_gpu(c, gid, w, outputs=("energy",))
        used = _used() - before
    assert used <= budget, used


def _crowded():
    """Modules under a canopy of 5 cm cells, 40 % of them holes, 16 suns: a
    128-texel tile is 20 cm of it, so most hold lit and shaded texels."""
    return S.make_canopy(31, map_res=4096, n=3, cells=60, n_steps=16)


def _reference(w, budget):
    """The results with the default budget, where the drawn tiles' records, of
    2 KB at least, take more than twice a quarter of `budget`."""
    with pv3d.Context(device=0, tile=128) as c:
        gid = pv3d.load_workload(c, w)
        big = run_gpu(c, gid, w, outputs=OUTS)
        c.evaluate(gid, n=w.n, map_res=w.map_res, profile=2)
        p = c.last_profile()
    assert (p["nonempty_tiles"] - p["sample_tiles"]) * (128 * 128 // 8) > budget // 2
    return big


def test_overflow_grows_the_pool():
    w, budget = _crowded(), 16 << 20
    big = _reference(w, budget)
    with pv3d.Context(device=0, tile=128, hbm_budget_bytes=budget) as c:
        gid = pv3d.load_workload(c, w)
        for _ in range(2):
            small = run_gpu(c, gid, w, outputs=OUTS)
            for k in OUTS:
                np.testing.assert_array_equal(small[k], big[k], err_msg=k)


def test_overflow_restarts_served_requests():
    import torch
    w, budget = _crowded(), 16 << 20
    big = _reference(w, budget)
    with pv3d.Context(device=0, tile=128, hbm_budget_bytes=budget, chunk_steps=16) as c:
        gid = pv3d.load_workload(c, w)
        rid, arrays = c.submit(gid, n=w.n, map_res=w.map_res, outputs=OUTS)
        assert c.poll(rid, timeout_ms=-1) == pv3d.PV3D_OK
        torch.cuda.synchronize()
        for k in OUTS:
            np.testing.assert_array_equal(arrays[k].cpu().numpy().view(big[k].dtype), big[k], err_msg=k)


def test_served_waves_use_their_scratch():
    """A served wave takes as many steps as wave_scratch_mb holds of what a step
    really takes: a byte a cell, 96 a module, 44 a tile and at most one record a
    tile."""
    w = S.make_tracker(seed=24, n=2, map_res=512, grid=(6, 5), terrain_n=48, spacing=3.0, n_pylons=1, step_h=1.0,
                       days=np.array([100, 280]))
    tiles = (512 // 64) ** 2
    step = w.gen.n_cells + 96 * w.gen.n_modules + tiles * (44 + 16 * (64 * 64 // 128 + 8)) + 512
    steps = w.sun.n_steps
    per_wave = (1 << 20) // step
    assert 2 <= per_wave < steps
    with pv3d.Context(device=0, tile=64, wave_scratch_mb=1) as c:
        gid = pv3d.load_workload(c, w)
        rid, got = c.submit(gid, n=w.n, map_res=w.map_res, outputs=("energy",))
        assert c.poll(rid, timeout_ms=-1) == pv3d.PV3D_OK
    assert got["waves"] <= -(-steps // per_wave)
