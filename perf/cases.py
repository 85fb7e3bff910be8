"""The work that users of this library have it do, as measurable cases.

Every case is one pass through the public Python entry points on inputs that
are already on the GPU, with the handles (grids, network) that a program keeps
from one input to the next:

  solve   new capacities -> mf_solve -> both cuts and the flow value, for one
          2D (4- or 8-connected) or 3D (6-connected) grid;
  batch   the same for many uneven grids at once (mf_set_caps_batch,
          mf_solve_batch, mf_get_cuts_batch);
  warm    a 2D solve from the learned warm start: features, network inference,
          projection to a preflow, solve;
  train   one training step of the warm-start network.

Inputs follow the workloads of the package's generators: value-noise
intensities for 2D segmentation, gradient noise with Gaussian class
likelihoods for volumes, the synthetic networks of Sec. 7.1 of the paper.
They are built on the GPU from a seed.
"""
import math
import os
import random

import numpy as np
import torch

import paper_1109_1146_gb300 as pkg
from paper_1109_1146_gb300 import mf

_WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(pkg.__file__)), "weights", "warm_seg2d_1024_c4.npy")

# forward half-stencils (dx, dy, dz) of the connectivities (see include/mf.h)
_FWD = {4: ((1, 0, 0), (0, 1, 0)),
        8: ((1, 0, 0), (0, 1, 0), (1, 1, 0), (-1, 1, 0)),
        6: ((1, 0, 0), (0, 1, 0), (0, 0, 1))}
# displacements (dx, dy) of the Sec. 7.1 networks in the library's order
_PAPER = ((1, 0), (0, 1), (1, 2), (2, 1), (1, 3), (3, 1), (2, 3), (3, 2), (0, 2), (2, 0), (2, 2), (3, 3), (3, 4), (4, 2))


def _solve(name, x, y, z, conn, inputs, **kw):
    c = {"kind": "solve", "x": x, "y": y, "z": z, "conn": conn, "inputs": inputs, "tile": "", "graph_loop": 0,
         "relabel": 4, "partial": 0}
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small 2D grid: a tile of an interactive segmentation, all latency
        _solve("seg2d_64_c4", 64, 64, 1, 4, "seg"),
        # the 256x256 segmentation grid, the smallest of the named workloads
        _solve("seg2d_256_c4", 256, 256, 1, 4, "seg"),
        # an image of odd size, 8-connected: ragged edge tiles, rows that are not 16-byte aligned
        _solve("seg2d_637x419_c8", 637, 419, 1, 8, "seg"),
        # a one-megapixel image, 4-connected, library defaults
        _solve("seg2d_1024_c4", 1024, 1024, 1, 4, "seg"),
        # the 2048x2048 8-connected grid with 5% hard seeds, tuned schedule (period 8, graph loop)
        _solve("seg2d_2048_c8_hard", 2048, 2048, 1, 8, "seg_hard", graph_loop=1, relabel=8),
        # a small ragged volume
        _solve("vol3d_61x75x53", 61, 75, 53, 6, "vol"),
        # a 128^3 volume, the largest member of the uneven batches
        _solve("vol3d_128", 128, 128, 128, 6, "vol"),
        # a full-size volume of 1.0e8 voxels
        _solve("vol3d_512x512x384", 512, 512, 384, 6, "vol"),
        # many uneven 2D and 3D grids at once (the mix of the batched benchmark, an eighth of its size)
        {"name": "batch_48x2d_16x3d", "kind": "batch", "n2d": 48, "n3d": 16, "shapes": 0, "graph_loop": 1,
         "relabel": 4},
        # the paper's synthetic network at its default connectivity 8 (knight moves), strength 150
        _solve("synthetic_500_c8", 500, 500, 1, 108, "synthetic", strength=150),
        # a megapixel solve from the learned warm start
        {"name": "warm_1024_c4", "kind": "warm", "x": 1024, "y": 1024},
        # a training step of the warm-start network: 8 crops of 256x256, 4-connected (6 channels)
        {"name": "train_8x256_c4", "kind": "train", "batch": 8, "x": 256, "y": 256, "conn": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("2d", "3d", "batch", "synthetic", "warm", "train"), (8, 6, 2, 2, 1, 1))[0]
    if kind == "2d":
        conn = rng.choice((4, 8))
        x = _log_int(rng, 48, 2048)
        y = max(48, min(2048, int(x * rng.uniform(0.5, 2.0))))
        return _solve("", x, y, 1, conn, rng.choice(("seg", "seg_hard")), tile=rng.choice(("", "", "64x32", "64x64")),
                      graph_loop=rng.randint(0, 1), relabel=rng.choice((2, 4, 8)), partial=int(rng.random() < 0.2))
    if kind == "3d":
        x, y, z = (_log_int(rng, 24, 224) for _ in range(3))
        return _solve("", x, y, z, 6, "vol", tile=rng.choice(("", "", "32x4x4", "32x8x8")),
                      graph_loop=rng.randint(0, 1), relabel=rng.choice((2, 4, 8)), partial=int(rng.random() < 0.2))
    if kind == "batch":
        return {"kind": "batch", "n2d": _log_int(rng, 6, 64), "n3d": _log_int(rng, 2, 16),
                "shapes": rng.randrange(1, 1 << 20), "graph_loop": rng.randint(0, 1), "relabel": rng.choice((4, 8))}
    if kind == "synthetic":
        c = rng.choice((8, 8, 12, 20))
        x = _log_int(rng, 100, 500)
        return _solve("", x, max(100, min(500, int(x * rng.uniform(0.7, 1.4)))), 1, 100 + c, "synthetic",
                      strength=rng.choice((20, 150, 400)) * 8 // c, graph_loop=rng.randint(0, 1))
    if kind == "warm":
        return {"kind": "warm", "x": _log_int(rng, 200, 1500), "y": _log_int(rng, 200, 1500)}
    return {"kind": "train", "batch": rng.randint(2, 8), "x": rng.randint(64, 256), "y": rng.randint(64, 256),
            "conn": rng.choice((4, 8))}


# --- inputs ----------------------------------------------------------------------

def _gen(seed):
    return torch.Generator().manual_seed(seed % (1 << 62))


def _fade(t):
    return t * t * t * (t * (t * 6.0 - 15.0) + 10.0)


def _to_u8(v):
    lo, hi = v.min(), v.max()
    return torch.round((v - lo) * (255.0 / (hi - lo).clamp_min(1e-12))).to(torch.int64)


def _value_noise(x, y, g):
    """Intensities 0..255 [y, x]: four octaves of value noise, lattice pitch 32/16/8/4."""
    xs, ys = torch.arange(x, device="cuda"), torch.arange(y, device="cuda")
    acc, amp = torch.zeros((y, x), dtype=torch.float64, device="cuda"), 1.0
    for pitch in (32, 16, 8, 4):
        lat = torch.rand((y // pitch + 2, x // pitch + 2), generator=g, dtype=torch.float64).cuda()
        gx, gy = xs // pitch, ys // pitch
        wx, wy = _fade((xs % pitch) / pitch)[None, :].double(), _fade((ys % pitch) / pitch)[:, None].double()
        top = lat[gy][:, gx] + (lat[gy][:, gx + 1] - lat[gy][:, gx]) * wx
        bot = lat[gy + 1][:, gx] + (lat[gy + 1][:, gx + 1] - lat[gy + 1][:, gx]) * wx
        acc += amp * (top + (bot - top) * wy)
        amp *= 0.5
    return _to_u8(acc)


_GRADS = ((1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1), (-1, 0, -1),
          (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1))


def _gradient_noise(x, y, z, g):
    """Intensities 0..255 [z, y, x]: three octaves of gradient noise, lattice pitch 32/16/8."""
    grads = torch.tensor(_GRADS, dtype=torch.float32, device="cuda")
    acc, amp = torch.zeros((z, y, x), dtype=torch.float32, device="cuda"), 1.0
    xs, ys = torch.arange(x, device="cuda"), torch.arange(y, device="cuda")
    for pitch in (32, 16, 8):
        pick = torch.randint(0, 12, (z // pitch + 2, y // pitch + 2, x // pitch + 2), generator=g)
        lat = grads[pick.cuda()]
        gx, gy = xs // pitch, ys // pitch
        fx, fy = (xs % pitch).float()[None, None, :] / pitch, (ys % pitch).float()[None, :, None] / pitch
        wx, wy = _fade(fx), _fade(fy)
        for z0 in range(0, z, 64):
            zs = torch.arange(z0, min(z, z0 + 64), device="cuda")
            gz, fz = zs // pitch, (zs % pitch).float()[:, None, None] / pitch
            wz = _fade(fz)
            for cz in (0, 1):
                for cy in (0, 1):
                    rows = lat[gz + cz][:, gy + cy]
                    for cx in (0, 1):
                        q = rows[:, :, gx + cx]
                        dot = q[..., 0] * (fx - cx) + q[..., 1] * (fy - cy) + q[..., 2] * (fz - cz)
                        w = (wx if cx else 1 - wx) * (wy if cy else 1 - wy) * (wz if cz else 1 - wz)
                        acc[z0:z0 + len(zs)] += amp * dot * w
        amp *= 0.5
    return _to_u8(acc)


def _lut(f):
    return torch.tensor([math.floor(f(i) + 0.5) for i in range(256)], dtype=torch.int32, device="cuda")


def _links(i3, conn, scale, sigma):
    """nlink[h] from the intensity difference across the h-th forward offset, 0 outside the grid."""
    z, y, x = i3.shape
    out = torch.zeros((len(_FWD[conn]), z, y, x), dtype=torch.int32, device="cuda")
    for h, (dx, dy, dz) in enumerate(_FWD[conn]):
        lut = _lut(lambda d: scale * math.exp(-d * d / (2 * sigma * sigma)) / (math.sqrt(2) if dx and dy else 1))
        x0, x1 = max(0, -dx), x - max(0, dx)
        a = i3[:z - dz, :y - dy, x0:x1]
        b = i3[dz:, dy:, x0 + dx:x1 + dx]
        out[h, :z - dz, :y - dy, x0:x1] = lut[(a - b).abs()]
    return out.reshape(len(out), -1)


def _seg2d(x, y, conn, g, hard=0.0, mu_fg=170.0, mu_bg=80.0):
    i = _value_noise(x, y, g)
    cs, ct = _lut(lambda v: abs(v - mu_bg))[i], _lut(lambda v: abs(v - mu_fg))[i]
    if hard:
        pick = (torch.rand((y, x), generator=g) < hard).cuda()
        fg = i >= (mu_fg + mu_bg) / 2
        cs = torch.where(pick, torch.where(fg, 10 ** 6, 0), cs).int()
        ct = torch.where(pick, torch.where(fg, 0, 10 ** 6), ct).int()
    return cs.reshape(-1), ct.reshape(-1), _links(i[None], conn, 100.0, 20.0)


def _vol3d(x, y, z, g):
    i = _gradient_noise(x, y, z, g)
    const = math.log(30.0 * math.sqrt(2 * math.pi))
    cs = _lut(lambda v: 10 * (const + (v - 80.0) ** 2 / 1800.0))[i]
    ct = _lut(lambda v: 10 * (const + (v - 170.0) ** 2 / 1800.0))[i]
    return cs.reshape(-1), ct.reshape(-1), _links(i, 6, 50.0, 15.0)


def _synthetic(x, y, conn, strength, g):
    e = torch.randint(-500, 501, (x * y,), generator=g, dtype=torch.int32).cuda()
    nl = torch.zeros(((conn - 100) // 2, y, x), dtype=torch.int32, device="cuda")
    for h in range(len(nl)):
        dx, dy = _PAPER[h]
        nl[h, :y - dy, :x - dx] = strength
    return e.clamp_min(0), (-e).clamp_min(0), nl.reshape(len(nl), -1)


def _caps(c, g):
    if c["inputs"] == "vol":
        return _vol3d(c["x"], c["y"], c["z"], g)
    if c["inputs"] == "synthetic":
        return _synthetic(c["x"], c["y"], c["conn"], c["strength"], g)
    return _seg2d(c["x"], c["y"], c["conn"], g, hard=0.05 if c["inputs"] == "seg_hard" else 0.0)


def _batch_shapes(c):
    """Uneven shapes: 2D sides uniform in 64..1024, 3D sides uniform in 48..128."""
    r = random.Random(c["shapes"])
    return [(r.randint(64, 1024),) * 2 + (1,) for _ in range(c["n2d"])] + [
        (r.randint(48, 128),) * 3 for _ in range(c["n3d"])]


def _warm_caps(c, seed):
    g = _gen(seed)
    mu_fg, mu_bg = (60.0 + 140.0 * torch.rand(2, generator=g, dtype=torch.float64)).tolist()
    return _seg2d(c["x"], c["y"], 4, g, mu_fg=mu_fg, mu_bg=mu_bg)


def _train_data(c, seed):
    """Features and solution flows of the size and spread the trainer sees (capacities / 100, flows of a solve)."""
    g = _gen(seed)
    shape = (c["batch"], c["conn"] + 2, c["y"], c["x"])
    x = torch.randint(0, 101, shape, generator=g).float().div(100).cuda()
    t = (torch.randn(shape, generator=g) * 0.25).cuda()
    return x, t


def _initial_params(ch, seed):
    """He-uniform weights and small biases, the library's parameter order."""
    g, out = _gen(seed + 1), []
    for co, ci in ((32, ch), (32, 32), (32, 32), (ch, 32)):
        out.append((2 * torch.rand(co * ci * 9, generator=g) - 1) * math.sqrt(6.0 / (9 * ci)))
        out.append((2 * torch.rand(co, generator=g) - 1) * 0.05)
    return torch.cat(out)


# --- the passes ------------------------------------------------------------------

def _outputs(n):
    return [torch.empty(n, dtype=torch.uint8, device="cuda") for _ in range(2)]


def prepare(case, seed):
    if case["kind"] == "solve":
        c, g = case, _gen(seed)
        tile = tuple(int(t) for t in c["tile"].split("x")) if c["tile"] else None
        grid = mf.Grid((c["x"], c["y"], c["z"]), c["conn"], tile=tile)
        opts = mf.default_opts(graph_loop=c["graph_loop"], global_relabel_period=c["relabel"],
                               partial_discharge=c["partial"])
        return {"kind": "solve", "grid": grid, "caps": _caps(c, g), "opts": opts, "cuts": _outputs(grid.n)}
    if case["kind"] == "batch":
        g = _gen(seed)
        grids, caps = [], []
        for x, y, z in _batch_shapes(case):
            grids.append(mf.Grid((x, y, z), 4 if z == 1 else 6))
            caps.append(_seg2d(x, y, 4, g) if z == 1 else _vol3d(x, y, z, g))
        opts = mf.default_opts(graph_loop=case["graph_loop"], global_relabel_period=case["relabel"])
        # the cuts of all grids in one buffer, each at a multiple of 256 bytes
        at = np.cumsum([0] + [(q.n + 255) // 256 * 256 for q in grids])
        flat = torch.zeros(int(at[-1]), dtype=torch.uint8, device="cuda")
        return {"kind": "batch", "grids": grids, "caps": caps, "opts": opts, "flat": flat,
                "cuts": [flat[a:a + q.n] for a, q in zip(at.tolist(), grids)]}
    if case["kind"] == "warm":
        grid = mf.Grid((case["x"], case["y"]), 4)
        net = mf.CNN(channels=6)
        net.load(_WEIGHTS)
        x = torch.empty((1, 6, case["y"], case["x"]), dtype=torch.float32, device="cuda")
        return {"kind": "warm", "grid": grid, "caps": _warm_caps(case, seed), "net": net, "x": x,
                "y": torch.empty_like(x), "cuts": _outputs(grid.n)}
    x, t = _train_data(case, seed)
    net = mf.CNN(channels=case["conn"] + 2)
    net.set_params(_initial_params(case["conn"] + 2, seed).numpy())
    return {"kind": "train", "net": net, "x": x, "t": t, "y": torch.empty_like(x), "dy": torch.empty_like(x)}


def _read(grid, cuts):
    return {"flow": grid.flow_value(), "smin": grid.get_cut(0, cuts[0]), "smax": grid.get_cut(1, cuts[1])}


def run(state):
    if state["kind"] == "solve":
        grid = state["grid"]
        grid.set_caps(*state["caps"])
        grid.solve(state["opts"])
        return _read(grid, state["cuts"])
    if state["kind"] == "batch":
        mf.set_caps_batch(state["grids"], state["caps"])
        mf.solve_batch(state["grids"], state["opts"])
        _, flows = mf.get_cuts_batch(state["grids"], 0, state["cuts"])
        return {"flows": np.array(flows, dtype=np.int64), "smin": state["flat"]}
    if state["kind"] == "warm":
        grid, x, y = state["grid"], state["x"], state["y"]
        grid.set_caps(*state["caps"])
        grid.warm_features(x)
        state["net"].infer(x, y)
        status, _ = grid.warm_start(y, check=False)
        grid.solve(mf.default_opts(warm_start=int(status == mf.MF_OK)))
        return dict(_read(grid, state["cuts"]), prediction=y)
    net = state["net"]
    net.forward(state["x"], state["y"])
    loss = net.mse(state["y"], state["t"], state["dy"])
    net.zero_grad()
    net.backward(state["x"], state["dy"])
    net.adam_step(lr=2e-3)
    return {"loss": loss, "y": state["y"], "grads": net.get_grads(), "params": net.get_params()}


def _network_flops(pixels, ch):
    return 2 * 9 * pixels * (2 * ch * 32 + 2 * 32 * 32)


def work(case):
    """Capacities read once, cuts written once; the network's products."""
    if case["kind"] == "batch":
        shapes = _batch_shapes(case)
        return {"bytes": sum(x * y * z * (4 * (2 + (2 if z == 1 else 3)) + 1) for x, y, z in shapes), "flops": 0}
    if case["kind"] == "solve":
        n, arcs = case["x"] * case["y"] * case["z"], case["conn"] % 100
        return {"bytes": n * (4 * (2 + arcs // 2) + 2), "flops": 0}
    n = case["x"] * case["y"]
    if case["kind"] == "warm":
        return {"bytes": n * (4 * 4 + 2 + 4 * 6), "flops": _network_flops(n, 6)}
    n, ch = n * case["batch"], case["conn"] + 2
    return {"bytes": 4 * n * ch * 3, "flops": 3 * _network_flops(n, ch) - 2 * 9 * n * ch * 32}


# --- 64-bit values ----------------------------------------------------------------

def _layers(params, ch):
    """[(weights rounded to BF16, bias)] in float64, leaves that take a gradient."""
    out, o = [], 0
    for co, ci in ((32, ch), (32, 32), (32, 32), (ch, 32)):
        w = params[o:o + co * ci * 9].reshape(co, ci, 3, 3)
        b = params[o + co * ci * 9:o + co * ci * 9 + co]
        o += co * ci * 9 + co
        out.append((w.bfloat16().double().requires_grad_(), b.double().requires_grad_()))
    return out


def _conv(h, w, b):
    """3x3 convolution with zero padding as nine matrix products, [n, y, x, c]."""
    n, y, x, _ = h.shape
    p = torch.nn.functional.pad(h, (0, 0, 1, 1, 1, 1))
    out = b.expand(n, y, x, len(b))
    for ky in range(3):
        for kx in range(3):
            out = out + p[:, ky:ky + y, kx:kx + x] @ w[:, :, ky, kx].t()
    return out


def _forward(x, layers):
    h = x.double().permute(0, 2, 3, 1)
    for i, (w, b) in enumerate(layers):
        h = _conv(h, w, b)
        if i < 3:
            h = torch.relu(h)
    return h.permute(0, 3, 1, 2)


def exact(case, seed):
    """Cuts and flow values are whole numbers; the network's outputs are given in float64 (weights rounded to BF16,
    as they enter every product)."""
    if case["kind"] == "warm":
        cs, ct, nl = (a.double() / 100 for a in _warm_caps(case, seed))
        y, x = case["y"], case["x"]
        cs, ct, right, down = cs.reshape(y, x), ct.reshape(y, x), nl[0].reshape(y, x), nl[1].reshape(y, x)
        left, up = torch.zeros_like(right), torch.zeros_like(down)
        left[:, 1:], up[1:] = right[:, :-1], down[:-1]
        with torch.no_grad():
            pred = _forward(torch.stack((cs, ct, right, left, down, up))[None],
                            _layers(torch.from_numpy(np.load(_WEIGHTS)).cuda(), 6))
        return {"flow": None, "smin": None, "smax": None, "prediction": pred}
    if case["kind"] == "train":
        ch = case["conn"] + 2
        x, t = _train_data(case, seed)
        params = _initial_params(ch, seed).cuda()
        layers = _layers(params, ch)
        y = _forward(x, layers)
        loss = ((y - t.double()) ** 2).mean()
        loss.backward()
        grads = torch.cat([q.grad.reshape(-1) for wb in layers for q in wb])
        after = params.double() - 2e-3 * grads / (grads.abs() + 1e-8)
        return {"loss": loss.item(), "y": y.detach(), "grads": grads.cpu().numpy(), "params": after.cpu().numpy()}
    return None
