"""The projection's colour rows and the adjoint's colour gradients with one view
and with the same camera twice, which read and write them by different routes
(each lane its own row; a warp's rows through shared memory): Gaussian counts at
the edges of a warp and a block, 3D / 4D borders inside a warp, time blocks."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import raster, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n3,n4", [(1, 0), (0, 1), (5, 27), (32, 1), (31, 64), (127, 1), (64, 65), (700, 333)])
@pytest.mark.parametrize("dtype,n_time", [(torch.float32, 0), (torch.float32, 2), (torch.bfloat16, 0), (torch.float16, 1)])
def test_one_view_and_the_same_view_twice(n3, n4, dtype, n_time):
    rng = np.random.default_rng(1000 * n3 + n4)
    c3, c4 = (np.concatenate([rng.uniform(-1, 1, (n, 2)), rng.uniform(2, 5, (n, 1))], 1) for n in (n3, n4))
    a = scenes.random_scene(rng, n3, n4, c3, c4).arrays()
    extra = rng.normal(0, 0.3, (n4, 16 * n_time, 3)).astype(np.float32)
    a["sh4"] = np.ascontiguousarray(np.concatenate([a["sh4"], extra], 1))
    G = raster.Gaussians.from_scene(scenes.Scene(**a), "cuda", dtype=dtype)
    view = scenes.identity_view(64, 48, 40.0, 0.3)
    N, out = n3 + n4, []
    dproj = torch.randn(12 * N, generator=torch.Generator().manual_seed(n3 + n4)).cuda()
    for V in (1, 2):
        R = raster.Rasterizer(n3, n4, [view] * V, sh_time=n_time)
        R.forward(G)
        R.dproj.zero_()
        R.dproj[: 12 * N] = dproj  # the second view adds zeros
        for g in R.grads.values():
            g.fill_(float("nan"))  # every row has to be written
        R.adjoint(G)
        torch.cuda.synchronize()
        R.check()
        out.append((R.rgb_depth.view(V, N, 4).clone(), {k: g.clone() for k, g in R.grads.items()}))
    (one, g1), (two, g2) = out
    assert torch.equal(two[0], one[0]) and torch.equal(two[1], one[0])
    for k in g1:
        # the same products (at most 8 FP32 roundings each), possibly contracted differently
        scale = float(g1[k].abs().max()) if g1[k].numel() else 0.0
        assert torch.isfinite(g1[k]).all() and torch.isfinite(g2[k]).all(), k
        if k.startswith("sh"):
            assert float((g1[k] - g2[k]).abs().max() if g1[k].numel() else 0.0) <= 1e-6 * scale, k
