"""Saturation heads of several windows: long lists of batches with at least two
super-tiles per SM.  The rows are written directly, wide footprints of a known
opacity over one half of a super-tile each, so that the two halves of a list end
in the window that the case says, or one of them never.  Every tile's list must be
a prefix of the list without culling, element by element, and the image, the
transmittance and the stops those of the uncut lists and of the radix path, bit
for bit."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import raster, scenes

pytestmark = pytest.mark.gpu

# (entries of the list, share that covers the upper half, opacity above, opacity below); a tile closes after about
# 9.25 / (0.94 opacity) entries of its half
LISTS = [
    (4097, 0.5, 0.04, 0.04),    # both in the first window
    (5000, 0.6, 0.02, 0.02),    # upper half in the second window, lower half in the third
    (5003, 0.35, 0.02, 0.02),   # the other way round, up to the end of the reach
    (6001, 0.6, 0.02, 0.005),   # upper half closes, the lower one stays open
    (4111, 0.5, 0.005, 0.03),   # upper half open, lower one in the second window
    (4096, 0.5, 0.02, 0.02),    # not a long list: one window, the rest in the tail
    (4500, 0.5, 0.0045, 0.006), # both open
    (700, 0.5, 0.05, 0.05),     # an ordinary list
]


def _rows(rng, lists, places, SX, TX, TY):
    """Rows of one view: list i in super-tile places[i]."""
    xy, co, rect, z = [], [], [], []
    for (n, upper, op_a, op_b), gs in zip(lists, places):
        sx, sy = gs % SX, gs // SX
        up = rng.uniform(size=n) < upper
        y0 = 8 * sy + np.where(up, 0, 4)
        rect.append(np.stack([np.full(n, 8 * sx), y0, np.full(n, min(8 * sx + 8, TX)), np.minimum(y0 + 4, TY)], 1))
        xy.append(np.stack([128 * sx + 64 + rng.uniform(-9, 9, n), 128 * sy + np.where(up, 32, 96) + rng.uniform(-9, 9, n)], 1))
        s2 = rng.uniform(210.0, 240.0, (2, n)) ** 2
        co.append(np.stack([1 / s2[0], np.zeros(n), 1 / s2[1], np.where(up, op_a, op_b) * rng.uniform(0.95, 1.05, n)], 1))
        z.append(rng.uniform(1.0, 20.0, n))
    return [np.concatenate(a).astype(d) for a, d in ((xy, np.float32), (co, np.float32), (rect, np.int32), (z, np.float32))]


def _load(R, views, rows):
    n = R.N
    out = [np.zeros((len(views) * n, k), d) for k, d in ((2, np.float32), (4, np.float32), (4, np.int32), (1, np.float32))]
    for v, r in enumerate(rows):
        m = len(r[0])
        for a, b in zip(out, r):
            a[v * n: v * n + m] = b.reshape(m, -1)
    xy, co, rect, z = out
    tiles = (rect[:, 2:] - rect[:, :2]).prod(-1).clip(0)
    assert (tiles >= 0).all()
    R.xy.copy_(torch.from_numpy(xy))
    R.conic_opacity.copy_(torch.from_numpy(co))
    R.rect.copy_(torch.from_numpy(rect))
    R.n_tiles.copy_(torch.from_numpy(tiles.astype(np.int32)))
    R.radius.copy_(R.n_tiles)
    rng = np.random.default_rng(1)
    rd = np.concatenate([rng.uniform(0, 1, (len(z), 3)).astype(np.float32), z], 1)
    R.rgb_depth.copy_(torch.from_numpy(rd))


def _run(R, cap, **options):
    R.set_options(**options)
    R.set_capacity(cap)
    R.status.zero_()
    R.bin_sort()
    R.composite()
    torch.cuda.synchronize()
    R.check()
    K = R.instances()
    return K, R.vals[:K].cpu().numpy(), R.ranges.view(-1, 2).cpu().numpy(), [x.clone() for x in (R.rgb, R.final_T, R.last)]


@pytest.mark.parametrize("V", [1, 3])
def test_heads_that_end_in_different_windows(V):
    rng = np.random.default_rng(V)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    SX = 20
    SY = -(-2 * sms // SX) if V == 1 else -(-sms // SX)
    # the last super-tiles hold three tile rows and five tile columns: their lower half lies outside the grid
    views = [scenes.identity_view(128 * SX - 48 - 5 * v, 128 * SY - 80 - 3 * v, 900.0, 0.5) for v in range(V)]
    TX = [(v.W + 15) // 16 for v in views]
    TY = [(v.H + 15) // 16 for v in views]
    rows = []
    for v in range(V):
        lists = LISTS if v == 0 else [LISTS[i] for i in rng.permutation(len(LISTS))[:4]]
        # the border's list covers the upper half only
        border = (4800, 1.0, 0.016, 0.016)
        inner = [int(y * SX + x) for y, x in zip(rng.permutation(SY - 1)[:len(lists)] if len(lists) < SY else
                                                  rng.integers(0, SY - 1, len(lists)), rng.permutation(SX - 1)[:len(lists)])]
        rows.append(_rows(rng, lists + [border], inner + [(SY - 1) * SX + 7], SX, TX[v], TY[v]))
    n = max(len(r[0]) for r in rows)
    R = raster.Rasterizer(n, 0, views, capacity=1 << 16)
    assert sum(-(-x // 8) * -(-y // 8) for x, y in zip(TX, TY)) >= 2 * sms
    _load(R, views, rows)
    whole = int(R.n_tiles.sum()) + 1
    K0, vals0, rg0, img0 = _run(R, whole, tile_sort=2, tile_cull=0)
    assert K0 == whole - 1
    S2 = 2 * sum(-(-x // 8) * -(-y // 8) for x, y in zip(TX, TY))
    _run(R, whole, tile_sort=2, tile_cull=1)
    need = int(R.n_needed.item())
    cut = None
    for cap in [max(need, 1024 * (k * sms - S2)) for k in (8, 40, 60)]:  # 32, 16 and 8 warps per segment
        K, vals, rg, img = _run(R, cap, tile_sort=2, tile_cull=1)
        assert K < K0
        for a, b in zip(img, img0):
            assert torch.equal(a, b)
        if cut is None:
            cut = (K, vals, rg)
            for t in range(R.total_tiles):
                m = rg[t, 1] - rg[t, 0]
                assert m <= rg0[t, 1] - rg0[t, 0]
                assert np.array_equal(vals[rg[t, 0]:rg[t, 1]], vals0[rg0[t, 0]:rg0[t, 0] + m])
        else:
            assert K == cut[0] and np.array_equal(vals, cut[1]) and np.array_equal(rg, cut[2])
    for a, b in zip(_run(R, whole, tile_sort=1, tile_cull=0)[3], img0):
        assert torch.equal(a, b)
    # the windows in which the first view's halves end: the position of a cut tile's last entry in its super-tile's list
    pos, depth = {}, R.rgb_depth[:, 3].cpu().numpy().view(np.uint32)
    K, vals, rg = cut
    first = 0
    ends = []
    for m, *_ in LISTS:
        ids = np.arange(first, first + m)
        first += m
        rank = np.empty(m, np.int64)
        rank[np.lexsort((ids, depth[ids]))] = np.arange(m)
        r = R.rect[int(ids[0])].cpu().numpy()
        got = []
        for row in (r[1] // 8 * 8, r[1] // 8 * 8 + 4):
            t = int(row * TX[0] + r[0] + 3)
            k, k0 = rg[t, 1] - rg[t, 0], rg0[t, 1] - rg0[t, 0]
            got.append(None if k == k0 else int(rank[vals[rg[t, 1] - 1] - ids[0]]) // 512)
        ends.append(got)
    assert ends[0] == [0, 0]
    assert ends[1] == [1, 2] or ends[1][0] < ends[1][1]
    assert ends[2][0] > ends[2][1] >= 1
    assert ends[3][0] is not None and ends[3][0] >= 1 and ends[3][1] is None
    assert ends[4][0] is None and ends[4][1] >= 1
    assert ends[5] == [None, None] and ends[6] == [None, None]
