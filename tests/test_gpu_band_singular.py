"""Bands of a tile (2 and 4 pixels per lane) and conics whose determinant is a few
rounding errors: its sign depends on how a compiler contracts a c - b b, and a band
may leave out a Gaussian only where no pixel of it can blend.  The images must be
the bits of the whole-tile walk."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import raster, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", range(4))
def test_nearly_singular_conics(seed):
    rng = np.random.default_rng(seed)
    n, W, H = 600, 61, 67
    TX, TY = (W + 15) // 16, (H + 15) // 16
    R = raster.Rasterizer(n, 0, [scenes.identity_view(W, H, 64.0, 0.5)], capacity=4 * n * TX * TY)
    a, c = rng.uniform(0.2, 1.6, (2, n)).astype(np.float32)
    b = np.sqrt(a.astype(np.float64) * c).astype(np.float32)
    for _ in range(seed):  # the determinant at zero, or some units in the last place of b above it
        b = np.nextafter(b, np.float32(0))
    b *= rng.choice([-1, 1], n).astype(np.float32)
    op = rng.uniform(0.02, 0.3, n).astype(np.float32)
    R.xy.copy_(torch.from_numpy(rng.uniform(0, 64, (n, 2)).astype(np.float32)))
    R.conic_opacity.copy_(torch.from_numpy(np.stack([a, b, c, op], 1)))
    R.rgb_depth.copy_(torch.from_numpy(np.concatenate([rng.uniform(0, 1, (n, 3)), rng.uniform(1, 9, (n, 1))], 1)
                                       .astype(np.float32)))
    R.rect.copy_(torch.tensor([0, 0, TX, TY], dtype=torch.int32))
    R.n_tiles.fill_(TX * TY)
    R.radius.fill_(1)
    out = []
    for ppl in (8, 4, 2):
        R.set_options(ppl_fwd=ppl, ppl_bwd=ppl, tile_cull=0)
        R.status.zero_()
        R.bin_sort()
        R.composite()
        torch.cuda.synchronize()
        R.check()
        assert R.instances() == n * TX * TY
        out.append((R.rgb.clone(), R.final_T.clone(), R.last.clone()))
    assert float(out[0][1].min()) < 0.5
    for o in out[1:]:
        assert all(torch.equal(x, y) for x, y in zip(o, out[0]))
