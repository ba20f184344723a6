"""Rows that lie on few depths (planes that face the camera): the depth bins are
then bounded by sampled entries in the order of the lists.  Element by element
against numpy's sort, at bins of both sizes, few visible rows, several views, depths
on both sides of the samples; and the time of a long list, which must not grow with
the square of its length."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import raster, scenes

from test_gpu_list_sort import _check

pytestmark = pytest.mark.gpu


def _z(kind, n, rng):
    z = {"equal": np.full(n, 7.25), "two": np.where(rng.uniform(size=n) < 0.3, 3.0, 9.0),
         "eight": 2.0 + rng.integers(0, 8, n), "plane": 5.0 + rng.normal(0, 1e-6, n),
         "plane and rest": np.where(rng.uniform(size=n) < 0.6, 5.0 + rng.normal(0, 1e-5, n), rng.uniform(1, 20, n)),
         "alternating": np.where(np.arange(n) % 2 == 0, 7.25, 9.0),
         # one long bin that the samples do not show, most of it one depth next to others
         "tenth": np.where(rng.uniform(size=n) < 0.13, np.where(rng.uniform(size=n) < 0.8, 5.0, rng.normal(5.0, 1e-4, n)),
                           rng.uniform(1, 20, n)),
         "runs": 1.0 + (np.arange(n) * 6 // n), "descending": 9.0 - (np.arange(n) * 5 // n)}[kind].astype(np.float32)
    few = rng.integers(0, n, 5)  # far outside, mostly unsampled
    z[few] = (1e-20, 0.5, 30.0, 1e20, 7.25)
    return z


KINDS = ["equal", "two", "eight", "plane", "plane and rest", "alternating", "tenth", "runs", "descending"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,visible", [(8193, 1.0), (30000, 1.0), (60000, 0.4), (60000, 0.05)])
def test_one_list(kind, n, visible):
    rng = np.random.default_rng(n)
    x0, y0 = rng.integers(0, 8, n), rng.integers(0, 8, n)
    _check([scenes.identity_view(128, 128, 128.0, 0.5)], n, np.stack([x0, y0, x0 + 1, y0 + 1], 1), _z(kind, n, rng),
           rng.uniform(size=n) < visible)


@pytest.mark.parametrize("kind", KINDS)
def test_few_bins_and_views_of_their_own(kind):
    """Few rows per super-tile (64 bins), nearly all of them in one; the views' depths differ."""
    rng = np.random.default_rng(5)
    views = [scenes.identity_view(W, H, 900.0, 0.5) for W, H in ((2000, 1600), (900, 700), (2000, 1600))]
    n = 9001
    rects, z = [], []
    for v, view in enumerate(views):
        TX, TY = (view.W + 15) // 16, (view.H + 15) // 16
        away = rng.uniform(size=n) < 0.1
        x0 = np.where(away, rng.integers(0, TX, n), 8 + rng.integers(0, 8, n))
        y0 = np.where(away, rng.integers(0, TY, n), 16 + rng.integers(0, 8, n))
        rects.append(np.stack([x0, y0, np.minimum(TX, x0 + 2), np.minimum(TY, y0 + 1)], 1))
        z.append(_z(kind if v != 1 else "plane and rest", n, rng) if v < 2 else rng.uniform(1, 20, n).astype(np.float32))
    _check(views, n, np.concatenate(rects), np.concatenate(z), rng.uniform(size=3 * n) < 0.9)


@pytest.mark.parametrize("kind", ["equal", "two", "alternating", "tenth", "plane and rest"])
def test_time_of_a_long_list(kind):
    n = 1_000_000
    rng = np.random.default_rng(0)
    R = raster.Rasterizer(n, 0, [scenes.identity_view(128, 128, 128.0, 0.5)], capacity=2 * n, keep_keys=False)
    R.set_options(tile_cull=0)
    x0, y0 = rng.integers(0, 8, n), rng.integers(0, 8, n)
    R.rect.copy_(torch.from_numpy(np.stack([x0, y0, x0 + 1, y0 + 1], 1).astype(np.int32)))
    R.n_tiles.fill_(1)

    def best(z):
        R.rgb_depth[:, 3] = torch.from_numpy(z).cuda()
        times = []
        for _ in range(12):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            R.bin_sort()
            e[1].record()
            torch.cuda.synchronize()
            R.check()
            times.append(e[0].elapsed_time(e[1]))
        return min(times)

    uniform = best(rng.uniform(1, 20, n).astype(np.float32))
    assert best(_z(kind, n, rng)) < 4 * uniform
