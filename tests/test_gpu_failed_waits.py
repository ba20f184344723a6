"""Bounded waits that run out at once (spin limit 0) while other blocks of the
same kernel have not begun, because another stream holds the SMs: the call
completes or reports the timeout, writes nothing outside its buffers, and the
next call is whole.  Binned and radix path."""
import pytest
import torch

from paper_2505_13215_gb300 import abi, raster, scenes

from test_gpu_capacity import guarded_sort

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [2, 1])
def test_waits_that_run_out(mode):
    scene, views = scenes.arc_scene(n=40000)
    G = raster.Gaussians.from_scene(scene, "cuda")
    R = raster.Rasterizer(G.n3, G.n4, views[:2])
    R.autotune_capacity(G)
    R.slice_project(G)
    busy, x = torch.cuda.Stream(), torch.randn(4096, 4096, device="cuda")
    abi.splat_set_tile_sort(mode)
    abi.splat_set_tile_cull(0)
    try:
        capacity = int(R.n_tiles.sum()) + 1
        code, _, _, good = guarded_sort(R, capacity)
        assert code == abi.SPLAT_OK
        K = int(good["n_instances"].inner.item())
        for _ in range(20):
            abi.splat_set_spin_limit(0)
            with torch.cuda.stream(busy):
                x = (x @ x).clamp(-1, 1)
            code, stage, _, bufs = guarded_sort(R, capacity)
            abi.splat_set_spin_limit(1 << 22)
            assert code in (abi.SPLAT_OK, abi.SPLAT_ERR_TIMEOUT)
            if code == abi.SPLAT_ERR_TIMEOUT:
                assert abi.STAGES[stage] in ("depth_sort", "scan", "duplicate", "tile_sort")
            assert all(b.intact() for b in bufs.values())
        code, _, _, bufs = guarded_sort(R, capacity)
        assert code == abi.SPLAT_OK
        for k in ("ranges", "n_instances"):
            assert torch.equal(bufs[k].inner, good[k].inner)
        for k in ("vals", "keys"):
            assert torch.equal(bufs[k].inner[:K], good[k].inner[:K])
    finally:
        abi.splat_set_spin_limit(1 << 22)
        abi.splat_set_tile_cull(1)
        abi.splat_set_tile_sort(0)
