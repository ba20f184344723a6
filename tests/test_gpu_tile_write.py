"""The writing pass on items without entries: most super-tiles are empty, and a
CTA goes from one straight to its next ticket.  The lists must equal numpy's
sort element by element, with 32, 16 and 8 warps per item (the choice follows
the capacity), after the cell passes and after the one-kernel lists."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import scenes

from test_gpu_list_sort import _check, _depths

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("items_per_sm", [8, 30, 60])
@pytest.mark.parametrize("n,W,H", [(9000, 3200, 2560), (3000, 1400, 1000)])
def test_empty_super_tiles_between_full_ones(n, W, H, items_per_sm):
    rng = np.random.default_rng(n)
    SX, SY = (W + 127) // 128, (H + 127) // 128
    full = rng.choice(SX * SY, max(3, SX * SY // 25), replace=False)  # one super-tile in 25 holds rows
    gs = full[rng.integers(0, len(full), n)]
    TX, TY = (W + 15) // 16, (H + 15) // 16
    x0 = np.minimum(8 * (gs % SX) + rng.integers(0, 8, n), TX - 1)
    y0 = np.minimum(8 * (gs // SX) + rng.integers(0, 8, n), TY - 1)
    x1 = np.minimum(np.minimum(x0 + rng.integers(1, 4, n), 8 * (x0 // 8) + 8), TX)
    y1 = np.minimum(np.minimum(y0 + rng.integers(1, 4, n), 8 * (y0 // 8) + 8), TY)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _check([scenes.identity_view(W, H, float(W), 0.5)], n, np.stack([x0, y0, x1, y1], 1), _depths("uniform", n, rng),
           rng.uniform(size=n) < 0.9, cap=1024 * (items_per_sm * sms - 2 * SX * SY))
