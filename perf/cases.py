"""The work whose speed is measured: cases of the framework's public entry
points over the sizes of its workloads (4 096 to 1 000 000 Gaussians, views of
96 to 1920 pixels a side, 1 to 16 views a launch, SH degrees 0 to 3).

A case is a dict of plain values; its "kind" says which part of the framework
it calls:

  direct  a short frame of plain FP32 direct optimisation, issued call by call
  view    one frame of the render-only path, replayed as a CUDA graph
  raster  projection, binning and compositing of a batch, and their reverse
  stage1  iterations of Stage 1 from the start of a frame, replayed as graphs
  stage2  the start of Stage 2 on a frame and one epoch of it
  loss    L1 + D-SSIM of a batch of views with its gradient
  cache   the transformation cache's query and its reverse through autograd

listed() gives the cases, draw() more of the same ranges, prepare() what a
program holds before the call, run() one pass, work() the bytes and
operations no implementation can do without, exact() the outputs in 64 bits.
"""
import math

import numpy as np
import torch

from paper_2403_01444_gb300 import engine, gs3, scenes
from paper_2403_01444_gb300.autograd import NTCContext, NTCTransform

DEV = "cuda"


def listed():
    return [
        # the smallest workload: 4K Gaussians in four thumbnails, FP32, no
        # graph: launches and latency
        {"name": "direct_small", "kind": "direct", "n": 4096, "deg": 1, "V": 4, "W": 128, "H": 96,
         "bin": 4, "iters": 5},
        # a viewer's frame of a small scene in a window of an odd size
        {"name": "view_odd", "kind": "view", "n": 48611, "deg": 2, "V": 1, "W": 477, "H": 363, "bin": 4},
        # a viewer's frame of the headline scene: cache query, SH rotation, render
        {"name": "view_hd", "kind": "view", "n": 250000, "deg": 3, "V": 1, "W": 1352, "H": 1014, "bin": 4},
        # render and reverse of the 50K-Gaussian workload's eight small views
        {"name": "raster_mid", "kind": "raster", "n": 50000, "deg": 2, "V": 8, "W": 480, "H": 360, "bin": 4},
        # render and reverse of one batch of the headline workload
        {"name": "raster_hd", "kind": "raster", "n": 250000, "deg": 3, "V": 4, "W": 1352, "H": 1014, "bin": 4},
        # Stage-1 training of the headline workload: one epoch (20 cameras in
        # five batches of four) from the start of a frame, mixed precision
        {"name": "stage1_hd", "kind": "stage1", "n": 250000, "deg": 3, "V": 4, "W": 1352, "H": 1014,
         "bin": 4, "iters": 5},
        # the largest workload: 1M Gaussians, 16 full-HD views in one launch
        {"name": "stage1_large", "kind": "stage1", "n": 1000000, "deg": 3, "V": 16, "W": 1920, "H": 1080,
         "bin": 4, "iters": 1},
        # Stage 2 of the 500K-Gaussian workload: spawn, one epoch (12 cameras
        # in three batches) over the fixed and about 3 000 added Gaussians
        {"name": "stage2_hd", "kind": "stage2", "n": 500000, "deg": 3, "V": 4, "W": 1280, "H": 720,
         "bin": 4, "iters": 3, "added": 3000},
        # the loss of one headline batch, and of one small view of odd width
        {"name": "loss_hd", "kind": "loss", "V": 4, "W": 1352, "H": 1014},
        {"name": "loss_odd", "kind": "loss", "V": 1, "W": 479, "H": 361},
        # the cache at the headline size in mixed precision, with the
        # gradients of a training batch (most Gaussians are seen by no view)
        {"name": "cache_bf16", "kind": "cache", "n": 250000, "bf16": True, "seen": 0.12},
        # the FP32 cache with every row's gradient, as when it is warmed up
        {"name": "cache_fp32", "kind": "cache", "n": 50000, "bf16": False, "seen": 1.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["direct", "view", "raster", "raster", "stage1", "stage2", "loss", "cache", "cache"])
    # widths spread over the range, half of them odd; heights of 1/2 to 1 width
    W = _log_int(rng, 97, 1920)
    W += (W + rng.randrange(2)) % 2 if W < 1920 else 0
    H = max(96, min(1080, int(W * rng.uniform(0.5, 1.0))))
    V = min(rng.choice([1, 2, 3, 4, 5, 8, 12, 16]), max(1, 4 * 1352 * 1014 // (W * H)))
    if kind == "loss":
        return {"kind": kind, "V": V, "W": W, "H": H}
    n = _log_int(rng, 4096, 500000)
    if kind == "cache":
        return {"kind": kind, "n": n, "bf16": rng.random() < 0.6, "seen": rng.choice([0.05, 0.12, 0.5, 1.0])}
    c = {"kind": kind, "n": n, "deg": rng.randrange(4), "V": 1 if kind == "view" else V, "W": W, "H": H,
         "bin": rng.choice([2, 4, 4, 4, 8])}
    if kind == "direct":
        c["n"] = _log_int(rng, 4096, 100000)
        c["iters"] = rng.randrange(2, 6)
    if kind == "stage1":
        c["iters"] = rng.randrange(1, 4)
    if kind == "stage2":
        c["iters"] = rng.randrange(1, 4)
        c["added"] = max(16, n // 150)
    return c


# ------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _rand(gen, *shape):
    return torch.rand(*shape, generator=gen, device=DEV)


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device=DEV)


def _gaussians(case, gen):
    """The distributions of the synthetic scenes: centres U[-1, 1]^3, log
    scales N(-3, 0.3), unit rotations, opacity logits N(0, 1), colours 0.5 +-
    0.4 with small higher SH bands."""
    n, K = case["n"], (case["deg"] + 1) ** 2
    mean = _rand(gen, n, 3) * 2 - 1
    quat = torch.nn.functional.normalize(_randn(gen, n, 4), dim=1)
    scale = torch.exp(_randn(gen, n, 3) * 0.3 - 3.0)
    opl = _randn(gen, n)
    sh = _randn(gen, n, K, 3) * 0.05
    sh[:, 0] = (_rand(gen, n, 3) * 2 - 1) * 1.4
    return gs3.Gaussians(mean, quat, scale, opl, sh, case["deg"])


def _cams(count, case):
    """Cameras on an arc of radius 4 around the scene, 60 degrees field of view."""
    return scenes.arc_cameras(count, case["W"], case["H"], (-60.0, 60.0) if count > 1 else (7.5, 7.5))


def _moved(g, gen):
    """The next frame's Gaussians: a smooth displacement of at most about 0.02 an axis."""
    ph = _rand(gen, 3) * 6.28
    return g.mean + 0.02 * torch.sin(3.0 * g.mean[:, [1, 2, 0]] + ph)


def _capacity(g, cams_dev, case):
    """Room for the pairs of a batch, with the margin a training program keeps."""
    r = engine.Rasterizer(g.n, case["V"], case["W"], case["H"], 1 << 20, bin=case["bin"])
    return max(1024, int(r.fit_capacity(g, cams_dev) * 2.0))


def _targets(g, gen, cams_dev, count, case):
    """The training views: renders of the moved Gaussians, V at a time."""
    V, W, H = case["V"], case["W"], case["H"]
    mean = _moved(g, gen)
    out = torch.empty(count, 3, H, W, device=DEV)
    for b in range(0, count, V):
        out[b:b + V] = engine.render_dev(g, gs3.camera_slice(cams_dev, b, V), V, W, H, mean, g.quat,
                                         bin=case["bin"])
    return out


def _cache_parameters(gen, entries):
    """A cache as its warm-up leaves it: outputs near the identity
    transformation (small translations, rotations near (1, 0, 0, 0))."""
    table = _randn(gen, entries, 2) * 0.05
    table[:, 0] += 0.5
    lim = lambda o, i: (_rand(gen, o, i) * 2 - 1) * math.sqrt(6.0 / i)
    w = [lim(64, 32), lim(64, 64), lim(7, 64)]
    w[2][0:3] *= 0.01
    w[2][3] = w[2][3].abs() + 1.0
    return table, w


def _ntc(gen, iters=engine.ITERS_PER_FRAME):
    grid = gs3.hashgrid()
    table, w = _cache_parameters(gen, gs3.ntc_hashgrid_entries(grid))
    return engine.NTC(table.cpu().numpy(), [x.cpu().numpy() for x in w], grid, gs3.GS_MLP_BF16, iters=iters)


def _image_grad(gen, case):
    V, W, H = case["V"], case["W"], case["H"]
    return _randn(gen, V, 3, H, W) / (3 * V * W * H)


def _loss_images(gen, case):
    """A render and its target: smooth images that differ a little, with flat regions."""
    V, W, H = case["V"], case["W"], case["H"]
    low = _rand(gen, V, 3, max(2, H // 24), max(2, W // 24))
    img = torch.nn.functional.interpolate(low, size=(H, W), mode="bilinear", align_corners=True)
    img = (img * 1.6 - 0.3).clamp_(0, 1).contiguous()
    target = (img + 0.03 * _randn(gen, V, 3, H, W)).clamp_(0, 1).contiguous()
    return img, target


def _cache_inputs(case, gen):
    n = case["n"]
    grid = gs3.hashgrid()
    table, w = _cache_parameters(gen, gs3.ntc_hashgrid_entries(grid))
    mean = _rand(gen, n, 3) * 2 - 1
    quat = torch.nn.functional.normalize(_randn(gen, n, 4), dim=1)
    seen = (_rand(gen, n, 1) < case["seen"]).float()
    d_mean = _randn(gen, n, 3) * 1e-2 * seen
    d_quat = _randn(gen, n, 4) * 1e-3 * seen
    return grid, table, torch.cat([x.reshape(-1) for x in w]), mean, quat, d_mean, d_quat


def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "loss":
        img, target = _loss_images(gen, case)
        return {"kind": kind, "loss": engine.Loss(case["V"], case["W"], case["H"]), "img": img, "target": target}
    if kind == "cache":
        grid, table, w, mean, quat, d_mean, d_quat = _cache_inputs(case, gen)
        ctx = NTCContext(grid, gs3.GS_MLP_BF16 if case["bf16"] else gs3.GS_MLP_FP32)
        return {"kind": kind, "ctx": ctx, "table": table.requires_grad_(), "w": w.requires_grad_(),
                "mean": mean, "quat": quat, "d_mean": d_mean, "d_quat": d_quat}
    V, W, H, S = case["V"], case["W"], case["H"], case["bin"]
    g = _gaussians(case, gen)
    if kind == "view":
        cd = gs3.cameras_to_device(_cams(V, case))
        r = engine.Renderer(g, _ntc(gen), V, W, H, _capacity(g, cd, case), bin=S)
        return {"kind": kind, "renderer": r, "cams": cd, "graph": r.capture(cd)}
    if kind == "raster":
        cd = gs3.cameras_to_device(_cams(V, case))
        r = engine.Rasterizer(g.n, V, W, H, 1 << 20, bin=S)
        r.fit_capacity(g, cd)
        return {"kind": kind, "raster": r, "g": g, "cams": cd, "d_img": _image_grad(gen, case)}
    if kind == "direct":
        cd = gs3.cameras_to_device(_cams(V, case))
        opt = engine.DirectOpt(g, V, W, H, _capacity(g, cd, case), bin=S)
        return {"kind": kind, "opt": opt, "g": g, "cams": cd, "iters": case["iters"],
                "target": _targets(g, gen, cd, V, case)}
    count = V * case["iters"]
    cams = gs3.cameras_to_device(_cams(count, case))
    target = _targets(g, gen, cams, count, case)
    batches = [(gs3.camera_slice(cams, b, V), target[b:b + V]) for b in range(0, count, V)]
    if kind == "stage1":
        ntc = _ntc(gen)
        warm = (ntc.init_table, ntc.init_mlp)
        st = engine.Stage1(g, ntc, V, W, H, _capacity(g, batches[0][0], case), bin=S)
        return {"kind": kind, "st": st, "warm": warm, "graphs": st.capture(batches), "keep": batches}
    st2 = engine.Stage2(g, V, W, H, capacity=2 * case["added"], bin=S)
    accum = torch.zeros(g.n, device=DEV)
    pick = torch.randperm(g.n, generator=gen, device=DEV)[:case["added"]]
    accum[pick] = 2 * engine.TAU_GRAD
    return {"kind": kind, "st2": st2, "batches": batches, "mean": _moved(g, gen), "accum": accum,
            "denom": torch.ones(g.n, dtype=torch.int32, device=DEV), "seed": seed}


# --------------------------------------------------------------------- pass
def run(s):
    kind = s["kind"]
    if kind == "direct":
        opt, g = s["opt"], s["g"]
        opt.mean.reset(g.mean)
        opt.quat.reset(g.quat)
        opt.state[4:].zero_()
        for _ in range(s["iters"]):
            loss = opt.step(s["cams"], s["target"])
        return {"loss": loss, "mean": opt.mean.p, "quat": opt.quat.p}
    if kind == "view":
        s["graph"].replay()
        r = s["renderer"]
        return {"img": r.raster.img, "mean": r.mean_t, "quat": r.quat_t}
    if kind == "raster":
        r = s["raster"]
        img = r.forward(s["g"], s["cams"])
        d_mean, d_quat = r.backward(s["g"], s["cams"], s["d_img"])
        return {"img": img, "d_mean": d_mean, "d_quat": d_quat, "pairs": r.d_count}
    if kind == "stage1":
        st = s["st"]
        st.ntc.reset_to(*s["warm"])
        st.reset_state()
        st.refresh_order()
        for graph in s["graphs"]:
            graph.replay()
        return {"loss": st.loss.d_loss, "table": st.ntc.table.p, "mlp": st.ntc.mlp.p}
    if kind == "stage2":
        st2 = s["st2"]
        st2.gen.manual_seed(s["seed"])
        st2.begin(s["mean"], st2.g.quat, s["accum"], s["denom"])
        n = st2.run(s["batches"], iters=len(s["batches"]))
        return {"n": n, "loss": st2.loss.d_loss, "rows": st2.rows[st2.cur][:n], "m": st2.m[st2.cur][:n]}
    if kind == "loss":
        loss = s["loss"]
        d_loss = loss(s["img"], s["target"])
        return {"loss": d_loss, "ssim": loss.d_ssim, "d_img": loss.d_img}
    mean_t, quat_t = NTCTransform.apply(s["table"], s["w"], s["mean"], s["quat"], s["ctx"])
    d_table, d_w = torch.autograd.grad([mean_t, quat_t], [s["table"], s["w"]], [s["d_mean"], s["d_quat"]])
    return {"mean": mean_t.detach(), "quat": quat_t.detach(), "d_table": d_table, "d_w": d_w}


# ---------------------------------------------------------------------- work
TABLE = 1647607            # rows of the hash table (16 levels, 2^17 rows a hashed level)
MLP = 64 * 32 + 64 * 64 + 7 * 64


def _blended(case):
    """Gaussians blended into a pixel, on average: those that reach it (the
    cloud fills about a (W / 2)^2 square; a footprint has sigma 0.05 / 4 fx,
    of which about three sigma count), until about 50 have hidden the rest."""
    W, H, n = case["W"], case["H"], case["n"]
    fx = W / (2 * math.tan(math.radians(30)))
    cloud = min(1.0, (2.2 * fx / 4) ** 2 / (W * H))
    reach = math.pi * (2.2 * 0.05 / 4 * fx) ** 2 * n / (2.2 * fx / 4) ** 2
    return cloud * min(50.0, 0.5 * reach)


def work(case):
    kind = case["kind"]
    if kind == "loss":
        px = 3 * case["V"] * case["W"] * case["H"]
        # two images in, a gradient out; five maps and three adjoint maps,
        # each through a separable window of 11 taps
        return {"bytes": 12 * px, "flops": px * 8 * 2 * 11 * 2}
    if kind == "cache":
        n = case["n"]
        seen = n * case["seen"]
        table = 4 * TABLE + 8 * TABLE if case["bf16"] else 16 * TABLE   # FP16 or FP32 in, FP32 gradient out
        return {"bytes": table + n * (28 + 28) + seen * 28 + 8 * MLP,
                "flops": n * (16 * 8 * 4 + 2 * MLP) + seen * (16 * 8 * 4 + 4 * MLP)}
    n, V, W, H = case["n"], case["V"], case["W"], case["H"]
    K = (case["deg"] + 1) ** 2
    px = V * W * H
    g_in = n * (44 + 12 * K)
    pairs = px * _blended(case)
    # a pair's quadratic form, exponential and blend: 21 operations; its reverse 59
    if kind == "view":
        return {"bytes": g_in + 4 * TABLE + 12 * px + n * 28, "flops": pairs * 21 + n * (1024 + 2 * MLP)}
    if kind == "raster":
        return {"bytes": g_in + 24 * px + 28 * n, "flops": pairs * 80}
    if kind == "direct":
        return {"bytes": case["iters"] * (g_in + 12 * px + 28 * n * 6), "flops": case["iters"] * pairs * 80}
    if kind == "stage1":
        # targets in; table and weights with their moments in and out
        step = 12 * px + (TABLE * 2 + MLP) * 4 * 6 + g_in
        return {"bytes": case["iters"] * step, "flops": case["iters"] * (pairs * 80 + px * 3 * 352 + n * 6 * MLP)}
    rows = case["added"] * (11 + 3 * K) * 4
    return {"bytes": case["iters"] * (g_in + 12 * px + 6 * rows), "flops": case["iters"] * (pairs * 80 + px * 3 * 352)}


# ------------------------------------------------------------- 64-bit results
def exact(case, seed):
    kind = case["kind"]
    gen = _gen(seed)
    if kind == "loss":
        img, target = _loss_images(gen, case)
        x = img.double().requires_grad_()
        loss, ssim = _loss64(x, target.double())
        (d_img,) = torch.autograd.grad(loss, x)
        return {"loss": loss.detach().reshape(1), "ssim": ssim.detach().reshape(1), "d_img": d_img}
    if kind == "cache":
        return _cache64(case, gen)
    # rendering in 64 bits visits every (Gaussian, pixel) pair of a tile in
    # plain torch: for the smaller scenes only
    tiles = case["V"] * -(-case["W"] // 16) * -(-case["H"] // 16)
    if kind == "raster" and tiles <= 6000 and case["n"] <= 60000:
        g = _gaussians(case, gen)
        cams = _cams(case["V"], case)
        d_img = _image_grad(gen, case).double()
        img, d_mean, d_quat = _render64(g, cams, case, d_img)
        return {"img": img, "d_mean": d_mean, "d_quat": d_quat, "pairs": None}
    return None


def _loss64(x, y, lam=0.2):
    """(1 - lam) mean|x - y| + lam (1 - SSIM), an 11-tap Gaussian window of sigma 1.5, zero padding."""
    t = torch.arange(11, dtype=torch.float64, device=x.device) - 5
    w = torch.exp(-t * t / 4.5)
    w = w / w.sum()
    V, C, H, W = x.shape

    def blur(a):
        a = a.reshape(V * C, 1, H, W)
        a = torch.nn.functional.pad(a, (5, 5, 5, 5))
        a = sum(w[k] * a[:, :, :, k:k + W] for k in range(11))
        a = sum(w[k] * a[:, :, k:k + H] for k in range(11))
        return a.reshape(V, C, H, W)

    mx, my = blur(x), blur(y)
    sxx, syy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = (((2 * mx * my + c1) * (2 * sxy + c2)) / ((mx * mx + my * my + c1) * (sxx + syy + c2))).mean()
    return (1 - lam) * (x - y).abs().mean() + lam * (1 - ssim), ssim


def _qmul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1)


def _cache64(case, gen):
    """Hash encoding, MLP and transformation with their gradients, in 64 bits."""
    grid, table, w, mean, quat, d_mean, d_quat = _cache_inputs(case, gen)
    table = table.double().requires_grad_()
    w = w.double().requires_grad_()
    m = mean.double()
    x01 = ((m + 1.5) / 3.0).clamp(0, 1)
    L, T = grid.levels, 1 << grid.log2_table
    b = math.exp((math.log(grid.n_max) - math.log(grid.n_min)) / (L - 1))
    off, feats = 0, []
    for l in range(L):
        N = int(math.floor(grid.n_min * b ** l + 1e-6))
        dense = (N + 1) ** 3 <= T
        p = x01 * N
        c = p.floor().clamp(max=N - 1)
        f = p - c
        c = c.long()
        acc = 0
        for corner in range(8):
            bit = [corner & 1, (corner >> 1) & 1, (corner >> 2) & 1]
            v = [c[:, k] + bit[k] for k in range(3)]
            if dense:
                h = v[0] + v[1] * (N + 1) + v[2] * (N + 1) ** 2
            else:
                h = (v[0] ^ (v[1] * 2654435761) ^ (v[2] * 805459861)) & (T - 1)
            wt = 1
            for k in range(3):
                wt = wt * (f[:, k] if bit[k] else 1 - f[:, k])
            acc = acc + wt[:, None] * table[off + h]
        feats.append(acc)
        off += (N + 1) ** 3 if dense else T
    e = torch.cat(feats, 1)
    w1, w2, w3 = w[:2048].reshape(64, 32), w[2048:6144].reshape(64, 64), w[6144:].reshape(7, 64)
    raw = torch.relu(torch.relu(e @ w1.T) @ w2.T) @ w3.T
    inside = (m.abs() <= 1.5).all(1, keepdim=True)
    norm = lambda q: q / q.norm(dim=1, keepdim=True).clamp(min=1e-12)
    qn = norm(quat.double())
    mean_t = torch.where(inside, m + raw[:, :3], m)
    quat_t = torch.where(inside, _qmul(qn, norm(raw[:, 3:])), qn)
    d_table, d_w = torch.autograd.grad([mean_t, quat_t], [table, w], [d_mean.double(), d_quat.double()])
    return {"mean": mean_t.detach(), "quat": quat_t.detach(), "d_table": d_table, "d_w": d_w}


def _sh_basis(deg, d):
    x, y, z = d.unbind(-1)
    o = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg > 0:
        c = math.sqrt(3 / (4 * math.pi))
        o += [-c * y, c * z, -c * x]
    if deg > 1:
        c = math.sqrt(15 / (4 * math.pi))
        o += [c * x * y, -c * y * z, math.sqrt(5 / (16 * math.pi)) * (2 * z * z - x * x - y * y), -c * x * z,
              c / 2 * (x * x - y * y)]
    if deg > 2:
        a, b = math.sqrt(35 / (32 * math.pi)), math.sqrt(105 / (4 * math.pi))
        e, f = math.sqrt(21 / (32 * math.pi)), math.sqrt(7 / (16 * math.pi))
        r = 4 * z * z - x * x - y * y
        o += [-a * y * (3 * x * x - y * y), b * x * y * z, -e * y * r,
              f * z * (2 * z * z - 3 * x * x - 3 * y * y), -e * x * r, b / 2 * z * (x * x - y * y),
              -a * x * (x * x - 3 * y * y)]
    return torch.stack(o, -1)


def _render64(g, cams, case, d_img):
    """The images of the batch and the gradients wrt means and rotations of
    sum(img * d_img), in 64 bits: per tile, its Gaussians by depth,
    blended front to back until the transmittance would fall below 1e-4."""
    W, H = case["W"], case["H"]
    tx, ty = -(-W // 16), -(-H // 16)
    mean = g.mean.double().requires_grad_()
    quat = g.quat.double().requires_grad_()
    scale, op, sh = g.scale.double(), torch.sigmoid(g.opacity_logit.double()), g.sh.double()
    imgs = torch.zeros(len(cams), 3, H, W, dtype=torch.float64, device=DEV)
    d_mean, d_quat = torch.zeros_like(mean), torch.zeros_like(quat)
    for v, c in enumerate(cams):
        vm = torch.from_numpy(np.asarray(c.viewmat, np.float64)).to(DEV)
        q = quat / quat.norm(dim=1, keepdim=True)
        qw, qx, qy, qz = q.unbind(-1)
        R = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                         2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                         2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)],
                        -1).reshape(-1, 3, 3)
        M = R * scale[:, None, :]
        t = mean @ vm[:, :3].T + vm[:, 3]
        z = t[:, 2]
        limx, limy = 1.3 * 0.5 * W / c.fx, 1.3 * 0.5 * H / c.fy
        ux, uy = (t[:, 0] / z).clamp(-limx, limx), (t[:, 1] / z).clamp(-limy, limy)
        zero = torch.zeros_like(z)
        J = torch.stack([c.fx / z, zero, -c.fx * ux / z, zero, c.fy / z, -c.fy * uy / z], -1).reshape(-1, 2, 3)
        P = J @ vm[:, :3] @ M
        cov = P @ P.transpose(1, 2) + 0.3 * torch.eye(2, dtype=torch.float64, device=DEV)
        a, b2, cc = cov[:, 0, 0], cov[:, 0, 1], cov[:, 1, 1]
        det = a * cc - b2 * b2
        A, B, C = cc / det, -b2 / det, a / det
        mid = 0.5 * (a + cc)
        r = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1)))).detach()
        u, w = c.fx * t[:, 0] / z + c.cx, c.fy * t[:, 1] / z + c.cy
        d = mean - torch.from_numpy(np.asarray(c.campos, np.float64)).to(DEV)
        Y = _sh_basis(case["deg"], d / d.norm(dim=1, keepdim=True))
        rgb = ((Y[:, :, None] * sh).sum(1) + 0.5).clamp(min=0)
        rec = torch.stack([u, w, A, B, C, rgb[:, 0], rgb[:, 1], rgb[:, 2]], -1)
        leaf = rec.detach().requires_grad_()
        ud, wd = u.detach(), w.detach()
        order = torch.argsort(z.detach())
        order = order[(z.detach()[order] > 0.2)]
        x0, x1 = ((ud - r) / 16).floor()[order], ((ud + r + 15) / 16).floor()[order]
        y0, y1 = ((wd - r) / 16).floor()[order], ((wd + r + 15) / 16).floor()[order]
        # the gradient wrt a record is a sum over tiles
        for j in range(ty):
            row = (y0 <= j) & (j < y1)
            orow, rx0, rx1 = order[row], x0[row], x1[row]
            for i in range(tx):
                ids = orow[(rx0 <= i) & (i < rx1)]
                px = torch.arange(16 * i, min(W, 16 * i + 16), device=DEV)
                py = torch.arange(16 * j, min(H, 16 * j + 16), device=DEV)
                if ids.numel() == 0:
                    continue
                e = leaf[ids]
                X = (px.double() + 0.5).repeat(py.numel())
                Yp = (py.double() + 0.5).repeat_interleave(px.numel())
                dx, dy = X[None] - e[:, 0:1], Yp[None] - e[:, 1:2]
                power = -0.5 * (e[:, 2:3] * dx * dx + e[:, 4:5] * dy * dy) - e[:, 3:4] * dx * dy
                al = (op[ids][:, None] * torch.exp(power)).clamp(max=0.99)
                al = torch.where((power <= 0) & (al >= 1 / 255), al, torch.zeros_like(al))
                T = torch.cumprod(1 - al, 0)
                keep = T >= 1e-4
                before = torch.cat([torch.ones_like(T[:1]), T[:-1]], 0)
                col = torch.einsum("np,nc->cp", torch.where(keep, al * before, torch.zeros_like(al)), e[:, 5:8])
                col = col.reshape(3, py.numel(), px.numel())
                ys, xs = slice(16 * j, 16 * j + py.numel()), slice(16 * i, 16 * i + px.numel())
                imgs[v][:, ys, xs] = col.detach()
                (col * d_img[v][:, ys, xs]).sum().backward()
        gm, gq = torch.autograd.grad(rec, [mean, quat], leaf.grad)
        d_mean += gm
        d_quat += gq
    return imgs, d_mean.detach(), d_quat.detach()
