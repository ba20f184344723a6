"""The forward's groups of Gaussians and the choice of pixels per lane by the
number of tiles, where they can go wrong: lists shorter than a group, lists that
end inside one, pixels that saturate at its first, a middle or its last Gaussian,
opacities at the clamp, images of odd sizes.  Every variant must give the bits of
an FP32 walk in the kernels' own operation order (power terms, 2^-x and T as they
are staged), which is also what the other variants give; the image is compared
with the FP64 oracle by the parity tests."""
import numpy as np
import pytest
import torch

from paper_2505_13215_gb300 import raster, scenes

pytestmark = pytest.mark.gpu


def _stack(n, logit, seed, W=37, H=21, spread=0.0, scales=(-1.5, 0.5)):
    """n Gaussians (wide ones by default) behind one another in front of a small image."""
    rng = np.random.default_rng(seed)
    means = np.stack([rng.uniform(-spread, spread, n), rng.uniform(-spread, spread, n), 2.0 + 0.01 * np.arange(n)], 1)
    s = scenes.random_scene(rng, n, 0, means, np.zeros((0, 3)))
    s.log_scale3[:] = rng.uniform(*scales, (n, 3)).astype(np.float32)
    s.opacity3[:] = np.asarray(logit, np.float32)
    return s, [scenes.identity_view(W, H, 40.0, 0.5)]


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 31, 33, 66])
@pytest.mark.parametrize("logit", [-2.0, 0.5, 3.0, 9.0])
def test_groups_agree_with_single_steps(n, logit):
    _agree(*_stack(n, logit, 100 * n + int(10 * logit), spread=0.2))


@pytest.mark.parametrize("scales", [(-5.0, -3.5), (-3.5, -2.5), (-6.0, 0.5)])
def test_bands_leave_out_only_what_they_do_not_reach(scales):
    """Footprints smaller than a band of a tile, about a tile, and needles across it (nearly singular conics)."""
    _agree(*_stack(700, 2.0, 5, W=61, H=67, spread=1.2, scales=scales))


def _agree(scene, views):
    G = raster.Gaussians.from_scene(scene, "cuda")
    counters = torch.zeros(8, dtype=torch.int64, device="cuda")
    out = []
    # the statistics instantiation walks one Gaussian at a time
    for ppl, stats in ((8, counters.data_ptr()), (2, None), (4, None), (8, None), (0, None)):
        R = raster.Rasterizer(G.n3, G.n4, views)
        R.set_options(ppl_fwd=ppl, ppl_bwd=ppl, stats=stats)
        target = torch.full_like(R.rgb, 0.25)
        R.autotune_capacity(G)
        R.step(G, target)
        torch.cuda.synchronize()
        R.check()
        out.append((R.rgb.clone(), R.final_T.clone(), R.last.clone(), R.grads["sh3"].clone()))
    assert (out[0][1] < 1.0).any()
    for o in out[1:]:
        for a, b in zip(o[:3], out[0][:3]):
            assert torch.equal(a, b)
        # the same terms in another order: n additions of FP32 rounding each, far below 1e-5 of the norm
        assert float((o[3] - out[0][3]).norm()) <= 1e-5 * float(out[0][3].norm())
