"""The super-tile list sort of the binned path at the sizes and depth
distributions where it can go wrong: lists around the size a block sorts in
shared memory, units cut into parts, crowded buckets, equal depths, depths far
outside the sampled range, rows over many super-tiles.  The projected rows are
written directly; the tile lists must equal numpy's stable sort by (tile, depth
bits) in row order, element by element."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import abi, raster, scenes

pytestmark = pytest.mark.gpu


def _depths(kind, n, rng):
    z = rng.uniform(1.0, 20.0, n)
    if kind == "equal":
        z[:] = 7.25
    elif kind == "two":
        z = np.where(np.arange(n) % 3 == 0, 3.0, 9.0)
    elif kind == "steps":
        z = np.round(z * 4) / 4 + 0.25
    elif kind == "narrow":
        z = rng.uniform(200.0, 200.5, n)
    elif kind == "outliers":
        z[: max(1, n // 300)] = rng.uniform(1e-30, 1e30, max(1, n // 300))
    elif kind == "clustered":  # nearly all depths within a few hundred FP32 steps
        z = np.where(rng.uniform(size=n) < 0.9, np.float32(5.0) + rng.integers(0, 300, n) * 2.0 ** -21, z)
    return z.astype(np.float32)


def _check(views, n, rects, z, visible, cap=None):
    R = raster.Rasterizer(n, 0, views, capacity=cap or int(1024 + 2 * (rects[..., 2:] - rects[..., :2]).prod(-1).sum()))
    R.set_options(tile_sort=2, tile_cull=0)
    area = np.where(visible, (rects[..., 2] - rects[..., 0]) * (rects[..., 3] - rects[..., 1]), 0)
    R.rect.copy_(torch.from_numpy(rects.astype(np.int32)))
    R.n_tiles.copy_(torch.from_numpy(area.astype(np.int32)))
    R.radius.copy_(R.n_tiles)
    R.rgb_depth[:, 3] = torch.from_numpy(z).cuda()
    R.bin_sort()
    torch.cuda.synchronize()
    R.check("sort")
    tile, row = [], []
    for v, view in enumerate(views):
        TX, TY = (view.W + 15) // 16, (view.H + 15) // 16
        base = abi.splat_total_tiles(R.W[:v], R.H[:v]) if v else 0
        for r in range(v * n, (v + 1) * n):
            if not visible[r]:
                continue
            x0, y0, x1, y1 = rects[r]
            t = (np.arange(y0, y1)[:, None] * TX + np.arange(x0, x1)[None]).ravel() + base
            tile.append(t)
            row.append(np.full(t.shape, r))
    tile = np.concatenate(tile) if tile else np.zeros(0, np.int64)
    row = np.concatenate(row) if row else np.zeros(0, np.int64)
    order = np.lexsort((row, z.view(np.uint32)[row], tile))
    K = R.instances()
    assert K == len(order)
    assert np.array_equal(R.keys[:K].cpu().numpy(), tile[order])
    assert np.array_equal(R.vals[:K].cpu().numpy(), row[order])
    first = np.searchsorted(tile[order], np.arange(R.total_tiles))
    last = np.searchsorted(tile[order], np.arange(R.total_tiles), side="right")
    rg = R.ranges.view(-1, 2).cpu().numpy()
    some = last > first
    assert np.array_equal(rg[some, 0], first[some]) and np.array_equal(rg[some, 1], last[some])
    assert (rg[~some] == 0).all()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 511, 512, 513, 545, 1536, 1537, 2047, 2048, 2049, 4096, 4097, 5000])
def test_one_super_tile(n):
    rng = np.random.default_rng(n)
    views = [scenes.identity_view(128, 128, 128.0, 0.5)]
    x0, y0 = rng.integers(0, 8, n), rng.integers(0, 8, n)
    rects = np.stack([x0, y0, np.minimum(8, x0 + rng.integers(1, 4, n)), np.minimum(8, y0 + rng.integers(1, 4, n))], 1)
    visible = rng.uniform(size=n) < 0.9
    visible[0] = True
    _check(views, n, rects, _depths("uniform", n, rng), visible)


@pytest.mark.parametrize("kind", ["uniform", "equal", "two", "steps", "narrow", "outliers", "clustered"])
@pytest.mark.parametrize("n", [700, 9000, 40000])
def test_depth_distributions(kind, n):
    rng = np.random.default_rng(7 + n)
    views = [scenes.identity_view(200, 120, 128.0, 0.5)]
    x0, y0 = rng.integers(0, 13, n), rng.integers(0, 8, n)
    rects = np.stack([x0, y0, x0 + 1, y0 + 1], 1)
    _check(views, n, rects, _depths(kind, n, rng), np.ones(n, bool))


def test_rows_over_many_super_tiles_in_views_of_different_sizes():
    rng = np.random.default_rng(3)
    views = [scenes.identity_view(W, H, 200.0, 0.5) for W, H in ((900, 410), (1, 1), (129, 257))]
    n = 300
    rects, vis = [], []
    for view in views:
        TX, TY = (view.W + 15) // 16, (view.H + 15) // 16
        x0, y0 = rng.integers(0, TX, n), rng.integers(0, TY, n)
        big = rng.uniform(size=n) < 0.3
        x1 = np.where(big, TX, np.minimum(TX, x0 + 1))
        y1 = np.where(big, TY, np.minimum(TY, y0 + 1))
        rects.append(np.stack([np.where(big, 0, x0), np.where(big, 0, y0), x1, y1], 1))
        vis.append(rng.uniform(size=n) < 0.8)
    _check(views, n, np.concatenate(rects), _depths("uniform", 3 * n, rng), np.concatenate(vis))


def test_no_visible_row():
    views = [scenes.identity_view(64, 64, 64.0, 0.5)]
    _check(views, 300, np.zeros((300, 4), np.int64), np.zeros(300, np.float32), np.zeros(300, bool), cap=1000)
