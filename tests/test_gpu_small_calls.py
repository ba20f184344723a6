"""Calls with few rows, whose super-tile lists are sorted by one block each, and
the tile order that the tile ranges write when one block holds every tile: row
counts around the limit (beyond it, and with more super-tiles than SMs, the cell
passes run instead), crowded depths, several views, the capacity to the entry."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import abi, raster, scenes

from test_gpu_list_sort import _check, _depths

pytestmark = pytest.mark.gpu


def _rects(n, TX, TY, rng, most=4):
    x0, y0 = rng.integers(0, TX, n), rng.integers(0, TY, n)
    return np.stack([x0, y0, np.minimum(TX, x0 + rng.integers(1, most, n)),
                     np.minimum(TY, y0 + rng.integers(1, most, n))], 1)


@pytest.mark.parametrize("n", [1023, 1025, 7169, 8191, 8192, 8193])
@pytest.mark.parametrize("kind", ["uniform", "equal", "two", "clustered", "outliers"])
def test_one_view(n, kind):
    rng = np.random.default_rng(n)
    _check([scenes.identity_view(250, 130, 128.0, 0.5)], n, _rects(n, 16, 9, rng), _depths(kind, n, rng),
           rng.uniform(size=n) < 0.9)


@pytest.mark.parametrize("n,V", [(300, 3), (2730, 3), (2731, 3), (8192, 4), (8193, 4), (6554, 5)])
def test_several_views(n, V):
    rng = np.random.default_rng(n)
    sizes = ((300, 170), (64, 20), (129, 257), (16, 16), (200, 140))
    views = [scenes.identity_view(W, H, 200.0, 0.5) for W, H in sizes[:V]]
    rects = np.concatenate([_rects(n, (v.W + 15) // 16, (v.H + 15) // 16, rng, 12) for v in views])
    _check(views, n, rects, _depths("uniform", V * n, rng), rng.uniform(size=V * n) < 0.7)


@pytest.mark.parametrize("n", [511, 2047, 2048, 2049, 4097])
def test_more_super_tiles_than_sms(n):
    rng = np.random.default_rng(n)
    views = [scenes.identity_view(128, 128, 128.0, 0.5), scenes.identity_view(1920, 1800, 900.0, 0.5)]
    rects = np.concatenate([_rects(n, 8, 8, rng), _rects(n, 120, 113, rng)])
    visible = np.concatenate([np.ones(n, bool), rng.uniform(size=n) < 0.05])
    _check(views, n, rects, _depths("uniform", 2 * n, rng), visible)


@pytest.mark.parametrize("W,H", [(128, 128), (256, 256), (272, 256)])
def test_capacity_and_tile_order(W, H):
    rng = np.random.default_rng(W)
    n, TX, TY = 900, (W + 15) // 16, (H + 15) // 16
    rects = _rects(n, TX, TY, rng, 6)
    K = int((rects[:, 2:] - rects[:, :2]).prod(-1).sum())  # at least the super-tiles' entries
    R = raster.Rasterizer(n, 0, [scenes.identity_view(W, H, 128.0, 0.5)], capacity=K)
    R.set_options(tile_sort=2, tile_cull=0)
    R.rect.copy_(torch.from_numpy(rects.astype(np.int32)))
    R.n_tiles.fill_(1)
    R.rgb_depth[:, 3] = torch.from_numpy(_depths("uniform", n, rng)).cuda()
    for cap in (K, K - 1, 600, K):  # (600: below the super-tiles' entries as well)
        R.status.zero_()
        R.set_capacity(cap)
        R.bin_sort()
        torch.cuda.synchronize()
        if cap == K:
            R.check("sort")
            assert R.instances() == K
        else:
            assert R.read_status()[0] == abi.SPLAT_ERR_CAPACITY
    length = (R.ranges.view(-1, 2)[:, 1] - R.ranges.view(-1, 2)[:, 0]).cpu().numpy()
    order = R.tile_order.cpu().numpy()[: TX * TY]
    assert np.array_equal(np.sort(order), np.arange(TX * TY))
    got = length[order]
    e = np.where(got > 0, np.floor(np.log2(np.maximum(got, 1))), 0)
    cls = np.where(got > 0, 1 + 8 * e + np.floor((got / 2.0 ** e - 1) * 8), 0)  # eight classes per power of two
    assert (np.diff(cls) <= 0).all()


def test_warps_per_segment():
    """The tail's passes take 32, 16 or 8 warps per segment by the capacity; the lists are the same."""
    rng = np.random.default_rng(11)
    views = [scenes.identity_view(250, 130, 128.0, 0.5)]
    n = 9000
    rects, z, visible = _rects(n, 16, 9, rng), _depths("uniform", n, rng), rng.uniform(size=n) < 0.9
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    caps = [1024 * sms * k for k in (4, 20, 50)]
    for cap in caps:
        _check(views, n, rects, z, visible, cap=cap)
    # with culling and ended lists, on a scene of full lists
    scene, arc = scenes.arc_scene(n=30000)
    G, out = raster.Gaussians.from_scene(scene, "cuda"), []
    for cap in caps:
        R = raster.Rasterizer(G.n3, G.n4, arc[:1], capacity=cap)
        R.forward(G)
        torch.cuda.synchronize()
        R.check()
        K = R.instances()
        out.append((K, R.vals[:K].clone(), R.keys[:K].clone(), R.ranges.clone()))
    for o in out[1:]:
        assert o[0] == out[0][0] and all(torch.equal(a, b) for a, b in zip(o[1:], out[0][1:]))
