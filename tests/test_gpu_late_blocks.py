"""The one-kernel lists of small calls where they overflow their capacity while other
blocks of the kernel have not begun."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import abi, raster, scenes

from test_gpu_capacity import guarded_sort, super_list_total
from test_gpu_list_sort import _depths
from test_gpu_small_calls import _rects

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [1, 4])
def test_capacity_overflow_with_blocks_that_start_late(V):
    """The block of the last super-tile reports the overflow while others may not have begun (another stream holds
    the SMs): nothing is written past a buffer, the needed count is exact, and the next call is whole."""
    rng = np.random.default_rng(V)
    n, W, H = 4000, 1300 // V, 1300
    R = raster.Rasterizer(n, 0, [scenes.identity_view(W, H, 900.0, 0.5)] * V)
    TX, TY = (W + 15) // 16, (H + 15) // 16
    rects = np.concatenate([_rects(n, TX, TY, rng, 9) for _ in range(V)])
    R.rect.copy_(torch.from_numpy(rects.astype(np.int32)))
    R.n_tiles.fill_(1)
    R.rgb_depth[:, 3] = torch.from_numpy(_depths("uniform", V * n, rng)).cuda()
    need = super_list_total(R)
    busy, x = torch.cuda.Stream(), torch.randn(4096, 4096, device="cuda")
    abi.splat_set_tile_cull(0)
    try:
        for k in range(20):
            with torch.cuda.stream(busy):
                x = (x @ x).clamp(-1, 1)
            code, _, aux, bufs = guarded_sort(R, need - 1 - 40 * k)
            assert code == abi.SPLAT_ERR_CAPACITY and aux == need
            assert all(b.intact() for b in bufs.values())
        code, _, _, bufs = guarded_sort(R, int((rects[:, 2:] - rects[:, :2]).prod(-1).sum()))
        assert code == abi.SPLAT_OK and all(b.intact() for b in bufs.values())
        K = int(bufs["n_instances"].inner.item())
        assert K == int((rects[:, 2:] - rects[:, :2]).prod(-1).sum())
    finally:
        abi.splat_set_tile_cull(1)
