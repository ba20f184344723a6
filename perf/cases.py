"""Performance cases of the hybrid 3D-4D Gaussian rasterizer: what a program that uses the
package has it do, through raster.Rasterizer / GraphedStep / HybridRasterize and the fused Adam.

A case is a dict of plain values:
  op        "render"    cameras set, then Rasterizer.forward (a viewer, a test-set evaluation)
            "step"      cameras set, then Rasterizer.step: forward, L1 loss, backward (training)
            "graph"     the same step replayed as a CUDA graph (GraphedStep)
            "autograd"  HybridRasterize inside torch autograd, with a loss of the user's own
            "adam"      the fused Adam launch over both parameter sets
  scene     "frustum"   Gaussians filling the view frustum, cameras near the base camera
            "arc"       Gaussians in a cube, cameras on an arc around it
  n, frac4  Gaussians, and the share of them that is 4D
  views     cameras per call (one batch); `mixed`: odd views at half resolution
  W, H      image size of the full-resolution views
  dtype     storage of the parameters; sh_time: time frequencies of the 4D colour

Sizes are those of the paper's setting (1352x1014 video frames, about 300k Gaussians, batches of
4 views), of its full 2704x2028 frames, and of the repository's tests and bench.  Parameters follow
the distributions of scenes.py, drawn on the device.
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2505_13215_gb300 import abi, raster, scenes, train

FIELDS3, FIELDS4 = raster.FIELDS3, raster.FIELDS4
DTYPES = {"float32": torch.float32, "bfloat16": torch.bfloat16, "float16": torch.float16}
DEVICE = "cuda"


def _case(name, op, scene, n, frac4, views, W, H, dtype, mixed=False, sh_time=0):
    c = {"op": op, "scene": scene, "n": n, "frac4": frac4, "views": views, "W": W, "H": H, "dtype": dtype,
         "mixed": mixed, "sh_time": sh_time}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a preview or thumbnail, one camera per call: latency and launches
        _case("render_128_4k", "render", "frustum", 4096, 0.25, 1, 128, 128, "float32"),
        # half-resolution frame of an odd size, FP16 checkpoint, 3D-dominated scene
        _case("render_677x507_101k_f16", "render", "arc", 101_003, 0.1, 1, 677, 507, "float16"),
        # the paper's rendering setting: one 1352x1014 frame of a 300k-Gaussian video
        _case("render_1352_300k", "render", "frustum", 300_000, 1 / 3, 1, 1352, 1014, "float32"),
        # a full-resolution frame of a large scene
        _case("render_2704_1m_bf16", "render", "arc", 1_000_000, 0.4, 1, 2704, 2028, "bfloat16"),
        # the smallest training step
        _case("graph_128_4k", "graph", "frustum", 4096, 0.25, 1, 128, 128, "float32"),
        # odd image sizes, mixed resolutions, time-dependent colour: fine-tuning on crops
        _case("step_857x479_120k_t2", "step", "arc", 120_007, 0.5, 3, 857, 479, "float16", True, 2),
        # the paper's training step: 4 views of 1352x1014, 300k Gaussians, BF16 storage
        _case("graph_1352_300k_v4_bf16", "graph", "frustum", 300_000, 1 / 3, 4, 1352, 1014, "bfloat16"),
        # a user's own loss through autograd, one FP32 view
        _case("autograd_1352_300k", "autograd", "frustum", 300_000, 1 / 3, 1, 1352, 1014, "float32"),
        # multi-camera batch at mixed resolutions, FP32
        _case("graph_1352_500k_v8", "graph", "arc", 500_000, 0.3, 8, 1352, 1014, "float32", True),
        # the largest batch of views, small frames, cameras changing every step
        _case("step_676_200k_v16_bf16", "step", "arc", 200_000, 0.33, 16, 676, 507, "bfloat16"),
        # training at the datasets' full resolution
        _case("graph_2704_1m_v4_bf16", "graph", "arc", 1_000_000, 0.4, 4, 2704, 2028, "bfloat16"),
        # the optimizer of the training step
        _case("adam_300k_bf16", "adam", "arc", 300_000, 1 / 3, 1, 64, 64, "bfloat16"),
    ]


def draw(rng):
    """A case of the same ranges: image widths 128 to 2704 and 0.05 to 0.5 Gaussians per pixel (both log-uniform),
    odd sizes, 1 to 16 views as far as the batch stays below four full-resolution views of a million Gaussians."""
    op = rng.choice(["render", "render", "graph", "graph", "step", "autograd", "adam"])
    scene = rng.choice(["frustum", "arc"])
    W = int(round(math.exp(rng.uniform(math.log(128), math.log(2704)))))
    H = max(96, int(round(W * rng.uniform(0.5, 0.8))))
    n = int(min(1_000_000, max(1000, W * H * math.exp(rng.uniform(math.log(0.05), math.log(0.5))))))
    most = int(min(16, 4 * 2704 * 2028 / (W * H), 4_000_000 / n))
    views = 1 if op in ("autograd", "adam") else int(round(math.exp(rng.uniform(0.0, math.log(max(1, most))))))
    if op == "render":
        views = min(views, 4)
    dtype = "float32" if op == "autograd" else rng.choice(["float32", "bfloat16", "float16"])
    if op == "adam":
        W = H = 64
        n = int(round(math.exp(rng.uniform(math.log(4096), math.log(1_000_000)))))
    return _case(None, op, scene, n, rng.choice([0.1, 0.25, 1 / 3, 0.5, 1.0]), views, W, H, dtype,
                 views > 1 and rng.random() < 0.5, rng.choice([0, 0, 0, 1, 2]))


# -- inputs -------------------------------------------------------------------

def _params(case, seed):
    """The parameter tensors in storage precision, and (n3, n4)."""
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    n4 = int(round(case["n"] * case["frac4"]))
    n3 = case["n"] - n4

    def normal(mean, std, *shape):
        return torch.randn(shape, generator=g, device=DEVICE) * std + mean

    def uniform(lo, hi, *shape):
        return torch.rand(shape, generator=g, device=DEVICE) * (hi - lo) + lo

    def means(n):
        if case["scene"] == "arc":
            return uniform(-5.0, 5.0, n, 3)
        near, far = (2.0, 6.0) if case["W"] <= 256 else (1.0, 20.0)
        f = _focal(case)
        z = uniform(near, far, n)
        return torch.stack([uniform(-1.0, 1.0, n) * (case["W"] / (2 * f)) * z,
                            uniform(-1.0, 1.0, n) * (case["H"] / (2 * f)) * z, z], 1)

    def quats(n):
        q = normal(0.0, 1.0, n, 4)
        return q / q.norm(dim=1, keepdim=True)

    def colours(n, blocks):
        sh = normal(0.0, 0.1, n, 16 * blocks, 3)
        sh[:, 0] = normal(0.0, 1.0, n, 3)
        return sh

    log4 = normal(-3.0, 0.5, n4, 4)
    log4[:, 3] = normal(-2.0, 0.5, n4)
    t = {"mean3": means(n3), "log_scale3": normal(-3.0, 0.5, n3, 3), "quat3": quats(n3),
         "opacity3": normal(0.0, 1.0, n3), "sh3": colours(n3, 1),
         "mean4": torch.cat([means(n4), uniform(0.0, 1.0, n4, 1)], 1), "log_scale4": log4, "ql": quats(n4),
         "qr": quats(n4), "opacity4": normal(0.0, 1.0, n4), "sh4": colours(n4, case["sh_time"] + 1)}
    return {k: v.to(DTYPES[case["dtype"]]).contiguous() for k, v in t.items()}, n3, n4


def _focal(case):
    return 1460.0 / 1352.0 * case["W"] if case["W"] > 256 else float(case["W"])


def _cameras(case, seed):
    """One camera (and timestamp) per view of the batch."""
    rng = np.random.default_rng(seed)
    f, V = _focal(case), case["views"]
    out = []
    for v in range(V):
        s = 2 if case["mixed"] and v % 2 else 1
        W, H = (case["W"] + s - 1) // s, (case["H"] + s - 1) // s
        t = float(rng.integers(0, 300)) / 299.0
        if case["scene"] == "arc":
            ang = math.radians(rng.uniform(-60.0, 60.0))
            eye = np.array([11.0 * math.sin(ang), rng.uniform(-1.0, 1.0), -11.0 * math.cos(ang)])
            out.append(scenes.look_at_view(eye, np.zeros(3), W, H, f / s, t))
        else:
            base = scenes.identity_view(W, H, f / s, t)
            out.append(scenes.jittered_views(base, 2, int(rng.integers(1 << 30)))[1])
            out[-1].t = t
    return out


def _target(case, n, seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed + 7)
    return torch.rand((n,), generator=g, device=DEVICE)


def _adam_grads(case, params, seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed + 13)
    return {k: torch.randn(v.shape, generator=g, device=DEVICE) * 1e-4 for k, v in params.items()}


ADAM = {"lr3": [8e-4, 5e-3, 1e-3, 5e-2, 2.5e-3], "lr4": [8e-4, 5e-3, 1e-3, 1e-3, 5e-2, 2.5e-3],
        "lr_sh_rest": 1.25e-4, "beta1": 0.9, "beta2": 0.999, "eps": 1e-15}


def prepare(case, seed):
    params, n3, n4 = _params(case, seed)
    s = {"case": case}
    if case["op"] == "adam":
        # FP32 master values and moments, and the storage copy that the same launch writes
        master = raster.Gaussians({k: v.float() for k, v in params.items()}, n3, n4)
        store = master if case["dtype"] == "float32" else raster.Gaussians(params, n3, n4)
        s.update(master=master, store=store, s3=train.AdamState(master, FIELDS3), s4=train.AdamState(master, FIELDS4),
                 grads=_adam_grads(case, params, seed), status=torch.zeros(4, dtype=torch.int32, device=DEVICE), t=0)
        s["cg3"] = abi.splat_grads3(*[s["grads"][k].data_ptr() for k in FIELDS3])
        s["cg4"] = abi.splat_grads4(*[s["grads"][k].data_ptr() for k in FIELDS4])
        h = abi.splat_adam_hyper()
        for i, lr in enumerate(ADAM["lr3"]):
            h.lr3[i] = lr
        for i, lr in enumerate(ADAM["lr4"]):
            h.lr4[i] = lr
        h.lr_sh_rest, h.beta1, h.beta2, h.eps = (ADAM[k] for k in ("lr_sh_rest", "beta1", "beta2", "eps"))
        s["hyper"] = h
        return s
    views = _cameras(case, seed)
    G = raster.Gaussians(params, n3, n4)
    R = raster.Rasterizer(n3, n4, views, device=DEVICE, keep_keys=False, sh_time=case["sh_time"])
    R.autotune_capacity(G)
    s.update(G=G, R=R, views=views)
    if case["op"] != "render":
        s["target"] = _target(case, R.rgb.numel(), seed)
    if case["op"] == "graph":
        s["graph"] = raster.GraphedStep(R, G, s["target"])
    if case["op"] == "autograd":
        s["params"] = [params[k].requires_grad_(True) for k in FIELDS3 + FIELDS4]
    return s


def run(s):
    op = s["case"]["op"]
    if op == "adam":
        s["t"] += 1
        s["hyper"].step = s["t"]
        g3, g4 = s["store"].c_g3(), s["store"].c_g4()
        abi.check(abi.splat_adam_step(C.byref(s["hyper"]), C.byref(s["s3"].c), C.byref(s["cg3"]), C.byref(g3),
                                      C.byref(s["s4"].c), C.byref(s["cg4"]), C.byref(g4),
                                      C.c_void_p(s["status"].data_ptr()),
                                      C.c_void_p(torch.cuda.current_stream().cuda_stream)), "splat_adam_step")
        out = {"master": dict(s["master"].t), "m": {**s["s3"].m, **s["s4"].m}, "v": {**s["s3"].v, **s["s4"].v}}
        if s["store"] is not s["master"]:
            out["store"] = dict(s["store"].t)
        return out
    R, G = s["R"], s["G"]
    if op == "autograd":
        rgb = raster.HybridRasterize.apply(R, G, *s["params"])
        loss = 0.5 * (rgb - s["target"]).square().mean()
        grads = torch.autograd.grad(loss, s["params"])
        return {"rgb": rgb.detach(), "loss": loss.detach(), "grads": dict(zip(FIELDS3 + FIELDS4, grads))}
    if op == "graph":
        s["graph"].replay()
    else:
        R.set_views(s["views"])
        if op == "render":
            R.forward(G)
            return {"rgb": R.rgb, "final_T": R.final_T}
        R.step(G, s["target"])
    return {"rgb": R.rgb, "final_T": R.final_T, "loss": R.loss, "grads": dict(R.grads)}


# -- what one pass cannot do without -------------------------------------------

def work(case):
    n, e = case["n"], {"float32": 4}.get(case["dtype"], 2)
    n4 = int(round(n * case["frac4"]))
    values = (n - n4) * 59 + n4 * (65 + 48 * case["sh_time"])
    if case["op"] == "adam":
        # gradient read; master, m and v read and written; the storage copy written
        return {"bytes": values * (28.0 + (e if e == 2 else 0)), "flops": values * 14.0}
    pix = sum(v.W * v.H for v in _cameras(case, 0))
    # pairs blended per pixel: the Gaussians in front of saturation, or those that cover a pixel at all
    f, full = _focal(case), case["W"] * case["H"]
    inv_z2 = {"arc": 1 / 100.0}.get(case["scene"], 1 / 12.0 if case["W"] <= 256 else 1 / 20.0)
    seen = (n - n4) + 0.3 * n4
    area = 2 * math.pi * 1.7 * (f * f * 0.0041 * inv_z2 + 0.3)
    pairs = pix * min(90.0, seen * area / full)
    fwd = {"bytes": values * e + pix * 20.0, "flops": pairs * 14.0 + n * case["views"] * 300.0}
    if case["op"] == "render":
        return fwd
    # target read, image gradient used, parameter gradients written
    return {"bytes": fwd["bytes"] + values * 4.0 + pix * 32.0, "flops": fwd["flops"] + pairs * 30.0 + n * case["views"] * 600.0}


# -- the same results in 64 bits -------------------------------------------------

def _f32(x):
    return float(np.float32(x))


def _quat_rot(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    rows = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
            2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
            2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]
    return torch.stack(rows, 1).view(-1, 3, 3)


def _rot4(ql, qr):
    a, b, c, d = (ql / ql.norm(dim=1, keepdim=True)).unbind(1)
    p, q, r, s = (qr / qr.norm(dim=1, keepdim=True)).unbind(1)
    left = torch.stack([a, -b, -c, -d, b, a, -d, c, c, d, a, -b, d, -c, b, a], 1).view(-1, 4, 4)
    right = torch.stack([p, -q, -r, -s, q, p, s, -r, r, -s, p, q, s, r, -q, p], 1).view(-1, 4, 4)
    return left @ right


def _sh16(d):
    """Real spherical harmonics of degree 0 to 3 (Condon-Shortley phase, m = -l..l)."""
    x, y, z = d.unbind(1)
    pi = math.pi
    k1, k2, k3 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / (4 * pi)), math.sqrt(35 / (32 * pi))
    k21, k30, k32 = math.sqrt(21 / (32 * pi)), math.sqrt(7 / (16 * pi)), math.sqrt(105 / (16 * pi))
    return torch.stack([
        torch.full_like(x, math.sqrt(1 / (4 * pi))), -k1 * y, k1 * z, -k1 * x,
        k2 * x * y, -k2 * y * z, math.sqrt(5 / (16 * pi)) * (3 * z * z - 1), -k2 * x * z, k2 / 2 * (x * x - y * y),
        -k3 * y * (3 * x * x - y * y), 2 * k32 * x * y * z, -k21 * y * (5 * z * z - 1),
        k30 * z * (5 * z * z - 3), -k21 * x * (5 * z * z - 1), k32 * z * (x * x - y * y),
        -k3 * x * (x * x - 3 * y * y)], 1)


def _project64(p, view, sh_time):
    """Slicing, EWA projection and colour of all Gaussians, 4D first: the splat features [n, 9]
    (x, y, conic, opacity, colour), and depth, radius, visibility."""
    R4 = _rot4(p["ql"], p["qr"])
    M = R4 * p["log_scale4"].exp().unsqueeze(1)
    S = M @ M.transpose(1, 2)
    t = _f32(view.t)
    dt = t - p["mean4"][:, 3]
    s44 = S[:, 3, 3]
    mu4 = p["mean4"][:, :3] + S[:, :3, 3] * (dt / s44).unsqueeze(1)
    u = M[:, 3] / M[:, 3].norm(dim=1, keepdim=True)
    B = M[:, :3] - (M[:, :3] @ u.unsqueeze(2)) * u.unsqueeze(1)
    M3 = _quat_rot(p["quat3"]) * p["log_scale3"].exp().unsqueeze(1)
    mu = torch.cat([mu4, p["mean3"]])
    cov = torch.cat([B @ B.transpose(1, 2), M3 @ M3.transpose(1, 2)])
    op = torch.cat([torch.sigmoid(p["opacity4"]) * torch.exp(-0.5 * dt * dt / s44), torch.sigmoid(p["opacity3"])])
    Rv = torch.from_numpy(np.asarray(view.R, np.float32).astype(np.float64)).to(mu)
    Tv = torch.from_numpy(np.asarray(view.T, np.float32).astype(np.float64)).to(mu)
    fx, fy, cx, cy = _f32(view.fx), _f32(view.fy), _f32(view.cx), _f32(view.cy)
    xc = mu @ Rv.T + Tv
    z = xc[:, 2]
    ux, uy = xc[:, 0] / z, xc[:, 1] / z
    limx, limy = 1.3 * 0.5 * view.W / fx, 1.3 * 0.5 * view.H / fy
    zero = torch.zeros_like(z)
    J = torch.stack([fx / z, zero, -fx * ux.clamp(-limx, limx) / z, zero, fy / z, -fy * uy.clamp(-limy, limy) / z],
                    1).view(-1, 2, 3)
    Tm = J @ Rv
    C2 = Tm @ cov @ Tm.transpose(1, 2)
    a, b, c = C2[:, 0, 0] + 0.3, C2[:, 0, 1], C2[:, 1, 1] + 0.3
    det = a * c - b * b
    d = mu + (Rv.T @ Tv)
    Y = _sh16(d / d.norm(dim=1, keepdim=True))
    sh4 = p["sh4"].view(-1, sh_time + 1, 16, 3)
    w = torch.tensor([math.cos(2 * math.pi * k * t) for k in range(sh_time + 1)], dtype=mu.dtype, device=mu.device)
    sh = torch.cat([torch.einsum("nbkc,b->nkc", sh4, w), p["sh3"]])
    rgb = (torch.einsum("nkc,nk->nc", sh, Y) + 0.5).clamp_min(0.0)
    px, py = fx * ux + cx, fy * uy + cy
    feat = torch.cat([torch.stack([px, py, c / det, -b / det, a / det, op], 1), rgb], 1)
    with torch.no_grad():
        lam = 0.5 * (a + c) + (0.25 * (a - c) ** 2 + b * b).clamp_min(0.1).sqrt()
        rad = torch.ceil(3 * lam.sqrt())
        TX, TY = (view.W + 15) // 16, (view.H + 15) // 16
        rect = torch.stack([torch.floor((px - rad) / 16).clamp(0, TX), torch.floor((py - rad) / 16).clamp(0, TY),
                            torch.ceil((px + rad) / 16).clamp(0, TX), torch.ceil((py + rad) / 16).clamp(0, TY)], 1)
        rect = torch.nan_to_num(rect).long()
        seen = (z > _f32(view.z_near)) & (op >= 1 / 255) & (det > 0)
        seen &= (rect[:, 2] > rect[:, 0]) & (rect[:, 3] > rect[:, 1])
    return feat, z.detach(), rect, seen


def _tile_lists(z, rect, seen, TX):
    """Gaussian index of every (tile, Gaussian) pair, by tile, then FP32 depth, then index; first pair of each tile."""
    order = torch.nonzero(seen).squeeze(1)
    order = order[torch.sort(z[order].float(), stable=True).indices]
    r = rect[order]
    w = r[:, 2] - r[:, 0]
    cnt = w * (r[:, 3] - r[:, 1])
    k = torch.repeat_interleave(torch.arange(len(order), device=z.device), cnt)
    off = torch.arange(len(k), device=z.device) - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
    tile = (r[k, 1] + off // w[k]) * TX + r[k, 0] + off % w[k]
    tile, by = torch.sort(tile, stable=True)
    return order[k[by]], tile


def _blend64(f, px, py, T0):
    """Weights of the splats f [B, L, 9] at pixels px, py [B, P] behind transmittance T0: colour, and the
    transmittance; a pixel stops in front of the splat that would take it below 1e-4."""
    dx, dy = f[:, None, :, 0] - px[:, :, None], f[:, None, :, 1] - py[:, :, None]
    power = -0.5 * (f[:, None, :, 2] * dx * dx + f[:, None, :, 4] * dy * dy) - f[:, None, :, 3] * dx * dy
    al = (f[:, None, :, 5] * power.exp()).clamp_max(0.99)
    al = torch.where((power > 0) | (al < 1 / 255), torch.zeros_like(al), al)
    T = T0[:, :, None] * torch.cumprod(1 - al, 2)
    live = T >= 1e-4
    w = torch.where(live, al * (T / (1 - al)), torch.zeros_like(al))
    Tend = T0 * torch.where(live, 1 - al, torch.ones_like(al)).prod(2)
    return w @ f[:, :, 6:9], Tend, live[:, :, -1]


def _render64(feat, lists, tile_of, view, dL=None):
    """The image [3, H, W] and final transmittance [H, W]; with dL [3, H, W]: the gradient of feat instead."""
    dev, TX, TY = feat.device, (view.W + 15) // 16, (view.H + 15) // 16
    n_tiles = TX * TY
    count = torch.bincount(tile_of, minlength=n_tiles)
    start = count.cumsum(0) - count
    rgb = torch.zeros((n_tiles, 256, 3), dtype=feat.dtype, device=dev)
    Tf = torch.ones((n_tiles, 256), dtype=feat.dtype, device=dev)
    lane = torch.arange(256, device=dev)
    data = torch.cat([feat.detach(), torch.zeros((1, 9), dtype=feat.dtype, device=dev)])  # the last row: no splat
    ends = torch.zeros_like(count)
    by = torch.argsort(count)
    chunk, batch = 256, 1024
    span = torch.arange(chunk, device=dev)

    def pixels(t):
        return ((t % TX) * 16)[:, None] + lane % 16, ((t // TX) * 16)[:, None] + lane // 16

    def rows(t, k, m):
        at = k + torch.arange(m, device=dev)
        have = at[None] < count[t][:, None]
        idx = lists[(start[t][:, None] + at[None]).clamp_max(max(0, len(lists) - 1))]
        return torch.where(have, idx, torch.full_like(idx, len(data) - 1))

    for q in range(0, n_tiles, batch):
        t, k = by[q: q + batch], 0
        x, y = pixels(t)
        open_ = ((x < view.W) & (y < view.H))
        while len(t):
            keep = (count[t] > k) & open_.any(1)
            t, open_, x, y = t[keep], open_[keep], x[keep], y[keep]
            if not len(t):
                break
            c, T1, live = _blend64(data[rows(t, k, chunk)], x.to(data), y.to(data), Tf[t])
            rgb[t] += torch.where(open_[:, :, None], c, torch.zeros_like(c))
            Tf[t] = torch.where(open_, T1, Tf[t])
            open_ = open_ & live
            k += len(span)
            ends[t] = torch.minimum(count[t], torch.full_like(t, k))
    bg = torch.tensor([_f32(b) for b in view.bg], dtype=feat.dtype, device=dev)

    def image(v):
        v = v.view(TY, TX, 16, 16, -1).permute(4, 0, 2, 1, 3).reshape(v.shape[2], TY * 16, TX * 16)
        return v[:, : view.H, : view.W]

    if dL is None:
        return image(rgb + Tf[:, :, None] * bg), image(Tf[:, :, None])[0]
    g = torch.zeros((3, TY * 16, TX * 16), dtype=feat.dtype, device=dev)
    g[:, : view.H, : view.W] = dL
    g = g.view(3, TY, 16, TX, 16).permute(1, 3, 2, 4, 0).reshape(n_tiles, 256, 3)
    out = torch.zeros_like(data)
    by, q = torch.argsort(ends), 0
    lens = ends[by].tolist()
    while q < n_tiles:
        if lens[q] == 0:
            q += 1
            continue
        e = q + 1
        while e < n_tiles and (e + 1 - q) * lens[e] <= 1 << 18:
            e += 1
        t = by[q:e]
        idx = rows(t, 0, lens[e - 1])
        f = data[idx].requires_grad_(True)
        x, y = pixels(t)
        with torch.enable_grad():
            c, T1, _ = _blend64(f, x.to(data), y.to(data), torch.ones((len(t), 256), dtype=data.dtype, device=dev))
            got, = torch.autograd.grad(((c + T1[:, :, None] * bg) * g[t]).sum(), f)
        out.index_add_(0, idx.reshape(-1), got.reshape(-1, 9))
        q = e
    return out[:-1]


def _adam64(case, seed):
    params, n3, n4 = _params(case, seed)
    grads = _adam_grads(case, params, seed)
    b1, b2, eps = _f32(ADAM["beta1"]), _f32(ADAM["beta2"]), _f32(ADAM["eps"])
    out = {"master": {}, "m": {}, "v": {}}
    for fields, lrs in ((FIELDS3, ADAM["lr3"]), (FIELDS4, ADAM["lr4"])):
        for k, lr in zip(fields, lrs):
            g = grads[k].double()
            step = torch.full(g.shape[1:], _f32(lr), dtype=torch.float64, device=DEVICE)
            if k in ("sh3", "sh4"):
                step[1:] = _f32(ADAM["lr_sh_rest"])
            out["m"][k] = (1 - b1) * g
            out["v"][k] = (1 - b2) * g * g
            out["master"][k] = params[k].double() - step * g / (g.abs() + eps)
    return out


def exact(case, seed):
    """run()'s results in 64 bits, by the plain definition: every Gaussian whose rectangle holds a pixel's tile, in
    depth order; gradients by autograd."""
    if case["op"] == "adam":
        return _adam64(case, seed)
    views = _cameras(case, seed)
    pix = sum(v.W * v.H for v in views)
    stored, n3, n4 = _params(case, seed)
    grad = case["op"] != "render"
    p = {k: v.double().requires_grad_(grad) for k, v in stored.items()}
    target = _target(case, 3 * pix, seed).double() if grad else None
    rgb, Ts, loss, at = [], [], 0.0, 0
    for view in views:
        with torch.set_grad_enabled(grad):
            feat, z, rect, seen = _project64(p, view, case["sh_time"])
        lists, tile_of = _tile_lists(z, rect, seen, (view.W + 15) // 16)
        with torch.no_grad():
            img, T = _render64(feat, lists, tile_of, view)
        rgb.append(img.reshape(-1))
        Ts.append(T.reshape(-1))
        if grad:
            diff = img - target[at: at + img.numel()].view_as(img)
            own = case["op"] == "autograd"
            loss = loss + (0.5 * diff.square().sum() / (3 * pix) if own else diff.abs().sum())
            dL = (diff if own else torch.sign(diff)) / (3 * pix)
            g = _render64(feat, lists, tile_of, view, dL)
            ok = seen.unsqueeze(1)  # rows that are not drawn may hold values without a derivative
            torch.autograd.backward(torch.where(ok, feat, feat.detach()), torch.where(ok, g, torch.zeros_like(g)))
        at += img.numel()
    out = {"rgb": torch.cat(rgb), "final_T": torch.cat(Ts)}
    if grad:
        out["loss"] = loss if case["op"] == "autograd" else loss.reshape(1)
        out["grads"] = {k: v.grad for k, v in p.items()}
    if case["op"] == "autograd":
        del out["final_T"]
    return out
