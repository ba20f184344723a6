"""Lists of the widest and the tallest image: super-tile coordinates up to their
largest value, rows at the far edge and across the whole image."""
import numpy as np
import pytest

from paper_2505_13215_gb300 import scenes

from test_gpu_list_sort import _check, _depths

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [600, 9000])
@pytest.mark.parametrize("W,H", [(16384, 200), (200, 16384), (16384, 33)])
def test_largest_coordinates(W, H, n):
    rng = np.random.default_rng(n + H)
    TX, TY = (W + 15) // 16, (H + 15) // 16
    x0, y0 = TX - 1 - rng.integers(0, TX, n) // 4, TY - 1 - rng.integers(0, TY, n) // 4
    rects = np.stack([x0, y0, np.minimum(TX, x0 + rng.integers(1, 9, n)), np.minimum(TY, y0 + rng.integers(1, 9, n))], 1)
    rects[:5] = [0, 0, TX, TY]
    rects[5] = [TX - 1, TY - 1, TX, TY]
    _check([scenes.identity_view(W, H, 900.0, 0.5)], n, rects, _depths("uniform", n, rng), np.ones(n, bool))
