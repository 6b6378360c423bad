"""The timed workloads of the library: what a program that uses it has it do.

Every case goes through the public entry points (``Context.compute``,
``Context.compute_host``, ``Context.compute_banded`` and the band network's
``sgmf_bn_*`` calls).  Inputs are generated on the GPU from a seed: layered
planar scenes with blurred-noise texture, a rectified right view, and a sparse
beam-pattern LiDAR map, in the shapes of the scenes the tests and the benchmark
use (256 x 128 to 1920 x 1080 pixels, 64 to 256 disparities).
"""
from __future__ import annotations

import math

import torch

from paper_2504_05148_gb300 import sgmf as S

# ---- the cases ---------------------------------------------------------------


def _plain(name, W, H, D, n, **kw):
    c = {"name": name, "kind": "plain", "W": W, "H": H, "D": D, "n": n, "sweep": False, "census": 0, "paths": 8,
         "semidense": 1, "check": 0, "subpixel": 0, "p1": 10, "p2": 120}
    c.update(kw)
    return c


def listed():
    return [
        # a thumbnail pair, one at a time: launches and latency
        _plain("tiny_pair", 256, 128, 64, 1),
        # one camera of the driving shape, one pair per call: a control loop's latency
        _plain("kitti_pair", 1242, 375, 128, 1),
        # the same from pinned host memory and back, waiting for the result
        _plain("kitti_host_pair", 1242, 375, 128, 1, kind="host"),
        # a few cameras' pairs gathered into one call, as the request loop forms them
        _plain("kitti_batch8", 1242, 375, 128, 8),
        # offline throughput: a large batch with the cluster sweep (the benchmark's shape and choice)
        _plain("kitti_batch32", 1242, 375, 128, 32, sweep=True),
        # indoor robot cameras, a class of the mixed-size batch, with the cluster sweep
        _plain("indoor_batch12", 640, 480, 64, 12, sweep=True),
        # low-light 720p frames with the full 62-bit census at 192 disparities
        _plain("lowlight_batch4", 1280, 720, 192, 4, census=1),
        # full-HD frames over the whole disparity range: a few per call
        _plain("hd_batch4", 1920, 1080, 256, 4),
        # a ragged crop, disparities that are no lane multiple, path costs beyond a byte, sub-pixel output
        _plain("ragged_subpixel", 333, 217, 100, 3, p2=300, subpixel=1),
        # the cheaper variant of the method: 4 paths, no semidensification, left-right check only
        _plain("fourpath_stereo", 1242, 375, 128, 4, paths=4, semidense=0, check=1),
        # full-HD frames restricted to 64-wide disparity bands, with the cluster sweep
        _plain("banded_hd_batch8", 1920, 1080, 256, 8, kind="banded", band=64, sweep=True),
        # one layer of the band network in training: forward, data gradient, weight gradient
        {"name": "bandnet_layer", "kind": "net", "W": 311, "H": 94, "n": 16},
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["plain"] * 6 + ["host", "banded", "banded", "net"])
    if kind == "net":
        return {"kind": "net", "W": logint(40, 480), "H": logint(24, 270), "n": logint(1, 16)}
    while True:
        W, H, n = logint(64, 1920), logint(40, 1080), logint(1, 32)
        D = rng.randint(16, 256) if kind != "banded" else rng.randint(64, 256)
        band = 128 if kind == "banded" and D >= 128 and rng.random() < 0.3 else 64
        cells = n * W * H * (band if kind == "banded" else D)
        if 3e5 <= cells <= 6e8:
            break
    c = _plain("", W, H, D, n, kind=kind)
    del c["name"]
    c["census"] = int(rng.random() < 0.2)
    c["paths"] = 4 if rng.random() < 0.15 else 8
    c["semidense"] = int(rng.random() >= 0.15)
    c["check"] = rng.choice([0, 0, 0, 0, 1, 2])
    c["subpixel"] = int(kind != "banded" and rng.random() < 0.25)
    c["p2"] = rng.choice([120, 120, 120, 60, 300])
    # the cluster sweep where rows fit one cluster and the batch is large
    lim = 1280 if D > 128 and kind != "banded" else 1920
    c["sweep"] = bool(c["paths"] == 8 and n >= 8 and W <= lim and rng.random() < 0.7)
    if kind == "banded":
        c["band"] = band
    return c


# ---- inputs ---------------------------------------------------------------------


def _blur(t, sigma=1.5, radius=5):
    k = [math.exp(-0.5 * (i / sigma) ** 2) for i in range(-radius, radius + 1)]
    W, H = t.shape[2], t.shape[1]
    p = torch.nn.functional.pad(t, (radius, radius, radius, radius), mode="circular")
    h = sum(k[i] * p[:, :, i:i + W] for i in range(2 * radius + 1))
    return sum(k[i] * h[:, i:i + H, :] for i in range(2 * radius + 1)) / sum(k) ** 2


def _texture(g, n, H, W):
    t = _blur(torch.rand((n, H, W), generator=g, device="cuda") * 255.0)
    t = (t - t.mean(dim=(1, 2), keepdim=True)) / t.std(dim=(1, 2), keepdim=True).clamp_min(1e-6)
    return (127.5 + t * 51.0).clamp(0.0, 255.0)


def _scene(n, W, H, D, seed, beams=True):
    """left, right uint8, lidar float32 and the true disparity float32, (n, H, W) on the GPU."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    y = torch.arange(H, device=dev, dtype=torch.float32).view(1, H, 1)
    x = torch.arange(W, device=dev, dtype=torch.float32).view(1, 1, W)
    # a far layer, a ground plane below the horizon, and slanted objects in front
    d = 0.03 * D + (y - 0.4 * H).clamp_min(0.0) * (0.75 * D / max(1.0, 0.6 * H)) + 0.0 * x
    d = d.repeat(n, 1, 1)
    u = torch.rand((20, 7, n, 1, 1), generator=g, device=dev)
    for k in range(20):
        cx, cy = u[k, 0] * W, (0.25 + 0.7 * u[k, 1]) * H
        hw, hh = (0.015 + 0.07 * u[k, 2]) * W, (0.03 + 0.15 * u[k, 3]) * H
        base = (0.05 + 0.75 * u[k, 4]) * D
        plane = base + (x - cx) * (u[k, 5] - 0.5) * 0.1 + (y - cy) * (u[k, 6] - 0.5) * 0.1
        inside = ((x - cx).abs() <= hw) & ((y - cy).abs() <= hh)
        d = torch.where(inside & (plane > d), plane, d)
    d = d.clamp(0.0, D - 1.0)
    # the right view is the texture; the left view looks it up at x - d, and
    # its pixels hidden in the right view (a nearer one lands there) or off it take fresh texture
    right = _texture(g, n, H, W)
    xs = x - d
    x0 = xs.floor()
    f = xs - x0
    i0 = x0.long().clamp(0, W - 1)
    i1 = (x0.long() + 1).clamp(0, W - 1)
    left = right.gather(2, i0) * (1.0 - f) + right.gather(2, i1) * f
    near = torch.zeros_like(d).scatter_reduce(2, xs.round().long().clamp(0, W - 1), d, "amax")
    hidden = (xs < 0) | (near.gather(2, xs.round().long().clamp(0, W - 1)) > d + 1.5)
    left = torch.where(hidden, _texture(g, n, H, W), left)
    noise = torch.randn((2, n, H, W), generator=g, device=dev)
    left = (left + 2.0 * noise[0]).round().clamp(0, 255).to(torch.uint8)
    right = (right + 2.0 * noise[1]).round().clamp(0, 255).to(torch.uint8)
    # beams on rows of the lower 60 % (denser toward the horizon), 29 % of a
    # beam row's columns return, 1 % of the returns are wrong
    nb = min(64, max(4, H // 4))
    t = torch.arange(nb, device=dev, dtype=torch.float32) / nb
    rows = (0.4 * H + (t ** 1.5) * (0.6 * H - 1)).long().clamp(0, H - 1)
    on = torch.zeros(H, dtype=torch.bool, device=dev)
    on[rows] = True
    r = torch.rand((3, n, H, W), generator=g, device=dev)
    keep = on.view(1, H, 1) & (r[0] < 0.29)
    val = d + 0.3 * torch.randn((n, H, W), generator=g, device=dev)
    val = torch.where(r[1] < 0.01, r[2] * D, val)
    lidar = torch.where(keep, val.clamp_min(0.0), torch.zeros_like(val)).contiguous()
    return left.contiguous(), right.contiguous(), lidar, d


def _params(c):
    p = S.Params()
    p.p1, p.p2 = c["p1"], c["p2"]
    p.census, p.num_paths, p.semidense = c["census"], c["paths"], c["semidense"]
    p.consistency, p.subpixel = c["check"], c["subpixel"]
    return p


def _net_inputs(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n, h, w = c["n"], c["H"], c["W"]
    x = torch.randn((n, h, w, 32), generator=g, device="cuda").clamp_min(0.0).to(torch.bfloat16)
    dy = (torch.randn((n, h, w, 32), generator=g, device="cuda") * 0.05).to(torch.bfloat16)
    wt = (torch.randn((32, 3, 3, 32), generator=g, device="cuda") * math.sqrt(2.0 / 288.0)).to(torch.bfloat16)
    bias = torch.randn(32, generator=g, device="cuda") * 0.1
    return x, dy, wt, bias


def prepare(case, seed):
    if case["kind"] == "net":
        x, dy, wt, bias = _net_inputs(case, seed)
        st = {"case": case, "x": x, "dy": dy, "w": wt, "bias": bias}
        st["packed_f"] = torch.empty(32 * 288, dtype=torch.int16, device="cuda")
        st["packed_d"] = torch.empty_like(st["packed_f"])
        stream = torch.cuda.current_stream().cuda_stream
        S.sgmf_bn_pack(wt.data_ptr(), st["packed_f"].data_ptr(), st["packed_d"].data_ptr(), stream)
        st["y"], st["dx"] = torch.empty_like(x), torch.empty_like(x)
        st["dw"] = torch.zeros((32, 3, 3, 32), dtype=torch.float32, device="cuda")
        st["db"] = torch.zeros(32, dtype=torch.float32, device="cuda")
        st["err"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        return st
    W, H, D, n = case["W"], case["H"], case["D"], case["n"]
    left, right, lidar, d = _scene(n, W, H, D, seed)
    ctx = S.Context(W, H, D, _params(case), max_batch=n, band=case.get("band", 0))
    if case["sweep"]:
        S.sgmf_set_tuning(ctx.handle, 4, 128, 1)
    st = {"case": case, "ctx": ctx}
    if case["kind"] == "host":
        for k, t in (("left", left), ("right", right), ("lidar", lidar)):
            st[k] = t.cpu().pin_memory().numpy()
        st["out"] = torch.empty((n, H, W), dtype=torch.int16).pin_memory().numpy()
        return st
    ctx.set_stream(torch.cuda.current_stream())
    st.update(left=left, right=right, lidar=lidar, out=torch.empty((n, H, W), dtype=torch.int16, device="cuda"))
    if case["kind"] == "banded":
        # per 8 x 8 tile, the band centred on its disparities: what a band proposal gives
        th, tw = (H + 7) // 8, (W + 7) // 8
        p = torch.nn.functional.pad(d[:, None], (0, tw * 8 - W, 0, th * 8 - H), mode="replicate")
        hi = torch.nn.functional.max_pool2d(p, 8)[:, 0]
        lo = -torch.nn.functional.max_pool2d(-p, 8)[:, 0]
        start = (0.5 * (lo + hi)).round() - case["band"] // 2
        st["band_lo"] = start.clamp(0, D - case["band"]).to(torch.int16).contiguous()
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "net":
        n, h, w = case["n"], case["H"], case["W"]
        s = torch.cuda.current_stream().cuda_stream
        err = st["err"].data_ptr()
        st["dw"].zero_()
        st["db"].zero_()
        S.sgmf_bn_conv(n, h, w, st["x"].data_ptr(), st["packed_f"].data_ptr(), st["bias"].data_ptr(), True, None,
                       st["y"].data_ptr(), None, err, s)
        S.sgmf_bn_wgrad(n, h, w, st["x"].data_ptr(), st["dy"].data_ptr(), st["dw"].data_ptr(), st["db"].data_ptr(),
                        err, s)
        S.sgmf_bn_conv(n, h, w, st["dy"].data_ptr(), st["packed_d"].data_ptr(), None, False, st["x"].data_ptr(),
                       st["dx"].data_ptr(), None, err, s)
        return {"y": st["y"], "dx": st["dx"], "dw": st["dw"], "db": st["db"]}
    ctx = st["ctx"]
    if kind == "host":
        ctx.compute_host(st["left"], st["right"], st["lidar"], st["out"])
    elif kind == "banded":
        ctx.compute_banded(st["left"], st["right"], st["lidar"], st["band_lo"], st["out"])
    else:
        ctx.compute(st["left"], st["right"], st["lidar"], st["out"])
    return st["out"]


def work(case):
    """Each input read once, each output written once; the operations of the method itself.

    Matching: per cell 8 operations per path (two adds of P1, three mins, the
    cost's add, the minimum's subtraction and its running min), the path sum,
    two running minima of the winner search, the Hamming cost's two.  Network
    layer: three contractions of 288 x 32 per pixel.
    """
    if case["kind"] == "net":
        px = case["n"] * case["H"] * case["W"]
        return {"bytes": px * 32 * 2 * 4 + 2 * (32 * 288 * 2 + 32 * 4) + 32 * 288 * 4 + 32 * 4,
                "flops": 3 * 2 * 288 * 32 * px}
    px = case["n"] * case["H"] * case["W"]
    d = case.get("band", case["D"])
    return {"bytes": px * (1 + 1 + 4 + 2), "flops": px * d * (8 * case["paths"] + case["paths"] + 2 + 2)}


def exact(case, seed):
    """The network layer in 64 bits.  Disparities are whole numbers: no rounding to judge."""
    if case["kind"] != "net":
        return None
    x, dy, wt, bias = _net_inputs(case, seed)
    xd = x.double().permute(0, 3, 1, 2)
    gd = dy.double().permute(0, 3, 1, 2)
    wd = wt.double().permute(0, 3, 1, 2)                       # [co][ci][ky][kx]
    h, w = case["H"], case["W"]
    xp = torch.nn.functional.pad(xd, (1, 1, 1, 1))
    gp = torch.nn.functional.pad(gd, (1, 1, 1, 1))
    y = torch.zeros_like(xd)
    dx = torch.zeros_like(xd)
    dw = torch.zeros((32, 3, 3, 32), dtype=torch.float64, device=x.device)
    for ky in range(3):
        for kx in range(3):
            xs = xp[:, :, ky:ky + h, kx:kx + w]
            y += torch.einsum("nihw,oi->nohw", xs, wd[:, :, ky, kx])
            dx += torch.einsum("nohw,oi->nihw", gp[:, :, 2 - ky:2 - ky + h, 2 - kx:2 - kx + w], wd[:, :, ky, kx])
            dw[:, ky, kx, :] = torch.einsum("nohw,nihw->oi", gd, xs)
    y = (y + bias.double().view(1, -1, 1, 1)).clamp_min(0.0)
    dx = dx * (xd > 0)
    return {"y": y.permute(0, 2, 3, 1).contiguous(), "dx": dx.permute(0, 2, 3, 1).contiguous(), "dw": dw,
            "db": gd.sum(dim=(0, 2, 3))}
