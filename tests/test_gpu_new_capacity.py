"""A new capacity means new list buffers: compositing before the next sort shows the
background, and reads nothing of a buffer that no sort has written."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import raster, scenes

pytestmark = pytest.mark.gpu


def test_compositing_before_the_next_sort():
    scene, views = scenes.small_scene(seed=3, n3=600, n4=200)
    views[0].bg = np.array([0.25, 0.5, 0.75], np.float32)
    G = raster.Gaussians.from_scene(scene, "cuda")
    R = raster.Rasterizer(G.n3, G.n4, views)
    R.autotune_capacity(G)
    assert not R.ranges.any()  # the capacity was cut down
    R.forward(G)
    image = R.rgb.clone()
    assert R.ranges.any()
    R.set_capacity(2 * R.capacity)
    R.composite()
    assert torch.equal(R.image(0), torch.tensor([0.25, 0.5, 0.75], device="cuda")[:, None, None].expand(3, 128, 128))
    assert bool((R.final_T == 1).all())
    R.forward(G)
    torch.cuda.synchronize()
    R.check()
    assert torch.equal(R.rgb, image)
