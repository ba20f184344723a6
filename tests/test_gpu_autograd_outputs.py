"""Gradients that HybridRasterize returns: shape, type and values of every field with
padded 3D capacity, an empty 3D or 4D set and 16-bit storage, in tensors of their
own (a later backward pass does not change them)."""
import pytest
import torch

from paper_2505_13215_gb300 import raster, scenes

pytestmark = pytest.mark.gpu

FIELDS = raster.FIELDS3 + raster.FIELDS4


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("n3,n4,pad", [(300, 100, 0), (300, 100, 77), (0, 200, 0), (0, 200, 31), (200, 0, 5)])
def test_returned_gradients(n3, n4, pad, dtype):
    scene, views = scenes.small_scene(seed=n3 + pad, n3=n3, n4=n4)
    G = raster.Gaussians.from_scene(scene, "cuda", dtype=dtype, capacity3=n3 + pad)
    R = raster.Rasterizer(G.n3, G.n4, views)
    R.autotune_capacity(G)
    params = [G.t[k].requires_grad_(True) for k in FIELDS]
    torch.manual_seed(0)
    w = torch.randn_like(R.rgb), torch.randn_like(R.rgb)
    got = []
    for x in w:
        rgb = raster.HybridRasterize.apply(R, G, *params)
        g = torch.autograd.grad((rgb * x).sum(), params)
        got.append((g, [t.clone() for t in g], {k: R.grads[k].clone() for k in FIELDS}))
    for g, copies, own in got:
        for k, p, t, c in zip(FIELDS, params, g, copies):
            assert t.shape == p.shape and t.dtype == dtype and t.device == p.device
            n = G.n3 if k in raster.FIELDS3 else G.n4
            assert torch.equal(t, c)  # the first pass's are unchanged after the second
            assert torch.equal(t[:n], own[k].to(dtype)) and not t[n:].any()
            assert t.numel() == 0 or t.data_ptr() != R.grads[k].data_ptr()
    if n3:
        assert got[0][0][0].abs().sum() > 0 and not torch.equal(got[0][0][0], got[1][0][0])
