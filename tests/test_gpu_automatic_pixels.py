"""The automatic number of pixels per lane: that the process-wide setting can return
to it, and launches with tile counts on both sides of each of its limits."""
import pytest
import torch

from paper_2505_13215_gb300 import abi, raster, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def automatic():
    abi.splat_set_pixels_per_lane(0, 0)
    yield
    abi.splat_set_pixels_per_lane(0, 0)


def _scene(TX, TY, n=400):
    W, H = 16 * TX - 5, 16 * TY - 3
    view = scenes.identity_view(W, H, 0.6 * max(W, H), 0.5)
    scene, _ = scenes.small_scene(seed=TX, n3=n, n4=0)
    scene.mean3[:, 0] *= W / max(W, H)
    scene.mean3[:, 1] *= H / max(W, H)
    return raster.Gaussians.from_scene(scene, "cuda"), [view]


def _launches(R, target):
    """Kernels of the fused forward: a second one sums the loss where it has more than 512 units (bands of tiles)."""
    n0 = abi.lib().splat_launch_count()
    R.composite_l1(target)
    return abi.lib().splat_launch_count() - n0


def test_the_setting_returns_to_automatic():
    G, views = _scene(20, 10)  # 200 tiles: 800 units at 2 pixels per lane, 400 at 4, 200 at 8
    R = raster.Rasterizer(G.n3, G.n4, views)
    R.autotune_capacity(G)
    R.forward(G)  # lists in the buffers of the new capacity
    target = torch.zeros_like(R.rgb)
    assert _launches(R, target) == 2
    abi.splat_set_pixels_per_lane(8, 8)
    assert _launches(R, target) == 1
    abi.splat_set_pixels_per_lane(3, -1)  # ignored
    assert _launches(R, target) == 1
    abi.splat_set_pixels_per_lane(0, 0)
    assert _launches(R, target) == 2
    R.set_options(ppl_fwd=4)
    assert _launches(R, target) == 1
    R.set_options(ppl_fwd=0)
    assert _launches(R, target) == 2
    torch.cuda.synchronize()
    R.check()


@pytest.mark.parametrize("tiles_per_sm", [2, 4, 10, 40])
def test_both_sides_of_each_limit(tiles_per_sm):
    limit = tiles_per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    for lo, step in ((limit, -1), (limit + 1, 1)):
        tiles = lo
        while not any(tiles % k == 0 and tiles // k <= 1024 for k in range(2, 90)):
            tiles += step
        TY = max(k for k in range(2, 90) if tiles % k == 0 and tiles // k <= 1024)
        G, views = _scene(tiles // TY, TY)
        R = raster.Rasterizer(G.n3, G.n4, views)
        assert R.total_tiles == tiles
        target, out = torch.full_like(R.rgb, 0.25), []
        for ppl in (0, 2, 4, 8):
            R.set_options(ppl_fwd=ppl, ppl_bwd=ppl)
            R.autotune_capacity(G)
            R.step(G, target)
            torch.cuda.synchronize()
            R.check()
            out.append((R.rgb.clone(), R.final_T.clone(), R.last.clone(), R.grads["sh3"].clone()))
        assert (out[0][1] < 1.0).any()
        for o in out[1:]:
            assert all(torch.equal(a, b) for a, b in zip(o[:3], out[0][:3]))
            # the same terms in another order: n additions of FP32 rounding each, far below 1e-5 of the norm
            assert float((o[3] - out[0][3]).norm()) <= 1e-5 * float(out[0][3].norm())
