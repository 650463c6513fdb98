"""The work that users of the block renderer have it do: cameras over baked
city blocks (one thumbnail up to the 1080p three-LOD city, and batches of
views), ray batches (validation rays, training steps with their gradients, the
per-block MLP form, the regularisers) and the optimiser's side of a fit.

``exact`` restates the rendering method in 64 bits with plain torch: which
lattice samples a ray takes is decided by the documented FP32 sequence, every
value after that (coordinates, lookups, weights, MLPs, losses, gradients) is
FP64, from the features as the storage format rounds them."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2312_16457_gb300 import cow, synth, train

DEV = "cuda"
ERT = 1e-5       # early ray termination of the viewer and of validation renders
OCC_CELL, OCC_THRESH = 4, 0.01
HIDDEN = 16


def listed():
    return [
        # a preview of one block while a scene is put together; launch and ray latency are what it costs
        {"name": "view_thumb_fp32", "kind": "view", "M": 1, "levels": 1, "R": 64, "P": 256, "storage": "fp32",
         "bricks": False, "width": 128, "height": 128, "ert": 0.0, "n_freq": -1},
        # an embedded viewer window of odd size over a small scene with the smallest storage forms, odd resolutions
        {"name": "view_odd_fp8_bricks", "kind": "view", "M": 3, "levels": 1, "R": 97, "P": 389,
         "storage": "fp8_bf16d", "bricks": True, "width": 517, "height": 391, "ert": ERT, "n_freq": -1},
        # a viewer that keeps every block's own MLP (the paper's form, Eq. 5), half of a 1080p window
        {"name": "view_block_mlps_bf16", "kind": "view", "M": 4, "levels": 1, "R": 128, "P": 512, "storage": "bf16",
         "bricks": False, "width": 960, "height": 540, "ert": ERT, "n_freq": 4},
        # the oblique city view at 720p
        {"name": "view_720p_fp16", "kind": "view", "M": 4, "levels": 1, "R": 256, "P": 1024, "storage": "fp16",
         "bricks": False, "width": 1280, "height": 720, "ert": ERT, "n_freq": -1},
        # the headline frame: LOD selection and the 1080p aerial view of the three-level city
        {"name": "view_1080p_lod_bf16", "kind": "view", "M": 8, "levels": 3, "R": 256, "P": 1024, "storage": "bf16",
         "bricks": False, "width": 1920, "height": 1080, "ert": ERT, "n_freq": -1},
        # a render server: a dozen cameras of uneven size in one call
        {"name": "batch_12_views_bf16", "kind": "batch", "M": 8, "levels": 3, "R": 128, "P": 512, "storage": "bf16",
         "bricks": False, "views": 12, "ert": ERT},
        # validation: random rays of held-out images through sixteen blocks, BF16 grid and FP8 planes
        {"name": "rays_eval_mixed", "kind": "eval", "M": 4, "levels": 1, "R": 128, "P": 512, "storage": "bf16_fp8",
         "n_rays": 30001, "ert": ERT},
        # a training mini-batch through torch.autograd
        {"name": "train_autograd_4k_fp32", "kind": "autograd", "M": 2, "levels": 1, "R": 64, "P": 256,
         "storage": "fp32", "n_rays": 4096},
        # a regularised training step that renders from BF16 copies
        {"name": "train_reg_64k_bf16", "kind": "train", "M": 2, "levels": 1, "R": 128, "P": 512, "storage": "bf16",
         "n_rays": 65537, "reg": True},
        # the full-size training step (the fit workload of the benchmark)
        {"name": "train_1m_fp32", "kind": "train", "M": 2, "levels": 1, "R": 128, "P": 512, "storage": "fp32",
         "n_rays": 1 << 20, "reg": False},
        # a training step of the per-block MLP form
        {"name": "train_block_mlps_fp32", "kind": "train_block", "M": 2, "levels": 1, "R": 128, "P": 512,
         "storage": "fp32", "n_rays": 100003, "n_freq": 2},
        # what follows the gradients: Adam on every parameter, the re-pack of the render copies, and a thumbnail of them
        {"name": "optimise_bf16", "kind": "optimise", "M": 2, "levels": 1, "R": 128, "P": 512, "storage": "bf16",
         "width": 96, "height": 54},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "view", "batch", "eval", "autograd", "train", "train", "train_block",
                       "optimise"])
    R = _log_int(rng, 24, 160)
    case = {"kind": kind, "M": rng.randint(1, 4), "levels": 1, "R": R, "P": 4 * R + rng.randint(-9, 9),
            "storage": rng.choice(["fp32", "fp16", "bf16", "bf16_fp8", "fp8_bf16d", "fp8"])}
    if kind == "view":
        case.update(bricks=rng.random() < 0.3, width=_log_int(rng, 64, 1600), height=_log_int(rng, 48, 900),
                    ert=rng.choice([0.0, ERT]), n_freq=rng.choice([-1, -1, 0, 2, 4]))
    elif kind == "batch":
        case.update(M=rng.choice([2, 4, 8]), levels=2, R=_log_int(rng, 24, 96), bricks=rng.random() < 0.3,
                    views=rng.randint(2, 20), ert=ERT)
        case["P"] = 4 * case["R"] + rng.randint(-9, 9)
    elif kind == "eval":
        case.update(n_rays=_log_int(rng, 1000, 400000), ert=rng.choice([0.0, ERT]))
    else:
        case.update(M=rng.randint(1, 2), storage=rng.choice(["fp32", "fp32", "bf16", "fp16"]))
        if kind == "optimise":
            case.update(width=_log_int(rng, 48, 200), height=_log_int(rng, 32, 120))
        else:
            case["n_rays"] = _log_int(rng, 1000, 300000)
        if kind == "autograd":
            case["storage"] = "fp32"
            case["n_rays"] = min(case["n_rays"], 65536)
        if kind == "train":
            case["reg"] = rng.random() < 0.4
        if kind == "train_block":
            case["n_freq"] = rng.randint(0, 4)
    return case


# --------------------------------------------------------------------------
# inputs (plain torch, from the seed alone)


def _generator(*keys):
    g = torch.Generator(device=DEV)
    h = 17
    for k in keys:
        h = (h * 1000003 + int(k) + 1) % (1 << 62)
    g.manual_seed(h)
    return g


def _uniform(gen, shape, lo, hi):
    return torch.rand(shape, generator=gen, device=DEV) * (hi - lo) + lo


def _field(case, seed):
    """Gaussian blobs over the ground's lower half, a ground slab, and the
    frequencies of the seven colour and specular channels."""
    half = float(case["M"])
    rng = np.random.default_rng([int(seed) % (1 << 31), 11])
    n = max(8, int(round(2.0 * (2 * half) ** 2)))
    centres = rng.uniform((-half, -half, -1.0), (half, half, 0.0), size=(n, 3))
    radii = rng.uniform(0.1, 0.3, size=n)
    dirs = rng.normal(size=(7, 3))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    return centres, radii, dirs * rng.uniform(2.0, 6.0, size=(7, 1)), rng.uniform(0, 2 * math.pi, size=7)


def _bake(case, seed, field, key, lo, hi, R, P):
    """One block's FP32 master arrays: log-density of blobs and slab, smooth
    colour channels with per-vertex noise, small plane features."""
    centres, radii, omega, phase = field
    x, y, z = (torch.linspace(lo[a], hi[a], R, device=DEV) for a in range(3))
    near = [k for k in range(len(radii)) if all(lo[a] - 5 * radii[k] < centres[k][a] < hi[a] + 5 * radii[k]
                                                for a in range(3))]
    c = torch.tensor(centres[near].reshape(-1, 3), dtype=torch.float32, device=DEV)
    r2 = torch.tensor(2.0 * radii[near] ** 2, dtype=torch.float32, device=DEV)
    ex, ey, ez = (torch.exp(-(v[None, :] - c[:, a:a + 1]) ** 2 / r2[:, None]) for a, v in enumerate((x, y, z)))
    sigma = torch.zeros((R, R, R), device=DEV)
    for k in range(len(near)):
        sigma += 20.0 * (ez[k][:, None, None] * (ey[k][:, None] * ex[k][None, :])[None])
    sigma += torch.where(z < -0.8, 20.0, 0.0)[:, None, None]
    gen = _generator(seed, 1, key)
    grid = torch.empty((R, R, R, 8), device=DEV)
    grid[..., 0] = torch.log(torch.clamp(sigma, min=1e-4))
    del sigma
    noise = _uniform(gen, (R, R, R, 7), -0.5, 0.5)
    for ch in range(7):
        wx, wy, wz = (float(v) for v in omega[ch])
        arg = (wz * z + float(phase[ch]))[:, None, None] + ((wy * y)[:, None] + (wx * x)[None, :])[None]
        grid[..., 1 + ch] = 1.5 * torch.sin(arg) + noise[..., ch]
    planes = [_uniform(gen, (P, P, 8), -0.1, 0.1) for _ in range(3)]
    return grid, planes


def _scene(case, seed):
    """Blocks of side 2 over [-M, M]^2 x [-1, 1], `levels` levels merged 2x2,
    coarse levels first; the thresholds keep the near blocks fine."""
    field = _field(case, seed)
    half, blocks, index = float(case["M"]), [], {}
    for lev in range(case["levels"], 0, -1):
        m, s = case["M"] >> (lev - 1), 2.0 * (1 << (lev - 1))
        R, P = max(2, case["R"] >> (lev - 1)), max(2, case["P"] >> (lev - 1))
        for j in range(m):
            for i in range(m):
                lo = (-half + i * s, -half + j * s, -1.0)
                hi = (lo[0] + s, lo[1] + s, 1.0)
                grid, planes = _bake(case, seed, field, len(blocks), lo, hi, R, P)
                index[(lev, i, j)] = len(blocks)
                blocks.append(synth.Block(lo, hi, R, P, lev, index.get((lev + 1, i // 2, j // 2), -1), grid, planes))
    return blocks, [12.5, 16.5, 0.0]


def _mlp(seed):
    return torch.randn(499, generator=_generator(seed, 2), device=DEV) * 0.3


def _block_mlps(seed, n_blocks, n_freq):
    gen = _generator(seed, 3)
    n = 16 * (10 + 6 * n_freq) + 339
    return (torch.randn(n, generator=gen, device=DEV) * 0.3
            + torch.randn((n_blocks, n), generator=gen, device=DEV) * 0.1)


def _look_at(pos, target):
    pos, fwd = np.asarray(pos, np.float64), np.asarray(target, np.float64) - np.asarray(pos, np.float64)
    fwd /= np.linalg.norm(fwd)
    right = np.cross(fwd, (0.0, 0.0, 1.0))
    right /= np.linalg.norm(right)
    return np.stack([right, np.cross(right, fwd), -fwd, pos], axis=1)


def _cameras(case, seed):
    """The viewer's camera (oblique, over the scene's edge) or the server's
    aerial cameras; (c2w, width, height, vertical field of view)."""
    rng = np.random.default_rng([int(seed) % (1 << 31), 5])
    half = float(case["M"])
    if case["kind"] != "batch":
        jit = rng.uniform(-0.05, 0.05, size=3) * half
        pos = {1: (0.0, -2.5, 0.8), 8: (0.0, -13.0, 9.0)}.get(case["M"], (0.0, -1.625 * half, 1.5 * half))
        tgt = (0.0, 0.0, 0.0) if case["M"] == 1 else (0.0, 0.1 * half, -1.0)
        fov = 40.0 if case["M"] in (2, 3, 4) else 60.0
        return [(_look_at(np.asarray(pos) + jit, tgt), case["width"], case["height"], fov)]
    cams = []
    for k in range(case["views"]):
        w, h = ((640, 360), (1280, 720), (333, 251), (1920, 1080), (1280, 720))[k % 5]
        pitch, yaw = math.radians(rng.uniform(30.0, 60.0)), rng.uniform(0.0, 2 * math.pi)
        up = rng.uniform(0.5, 1.0) * half + 2.0
        tgt = np.array([rng.uniform(-0.6, 0.6) * half, rng.uniform(-0.6, 0.6) * half, -1.0])
        away = up / math.tan(pitch)
        cams.append((_look_at(tgt + np.array([-away * math.cos(yaw), -away * math.sin(yaw), up]), tgt), w, h, 60.0))
    return cams


def _rays(case, seed):
    """Rays from a sphere around the scene towards uniform points of its box,
    and a target colour for each."""
    gen, n, half = _generator(seed, 4), case["n_rays"], float(case["M"])
    v = torch.randn((n, 3), generator=gen, device=DEV).double()
    o = v / v.norm(dim=1, keepdim=True) * (1.5 * math.sqrt(8 * half * half + 4.0))
    tgt = torch.rand((n, 3), generator=gen, device=DEV).double() * 2 - 1
    d = tgt * torch.tensor([half, half, 1.0], device=DEV, dtype=torch.float64) - o
    return o.float(), (d / d.norm(dim=1, keepdim=True)).float(), torch.rand((n, 3), generator=gen, device=DEV)


REG_POINTS, REG_SPARSITY, REG_OPACITY = 1 << 14, 0.05, 0.001


def _reg_points(case, seed):
    half = float(case["M"])
    u = torch.rand((REG_POINTS, 3), generator=_generator(seed, 6), device=DEV) * 2 - 1
    return u * torch.tensor([half, half, 1.0], device=DEV)


def _moments(case, seed, blocks):
    """Gradients and Adam moments of a fit under way, per parameter tensor."""
    gen, out = _generator(seed, 7), []
    for b in blocks:
        for p in (b.grid, *b.planes):
            out.append((torch.randn(p.shape, generator=gen, device=DEV) * 1e-3,
                        torch.randn(p.shape, generator=gen, device=DEV) * 1e-3,
                        torch.rand(p.shape, generator=gen, device=DEV) * 1e-6))
    return out


# --------------------------------------------------------------------------
# the cases through the framework


def prepare(case, seed):
    kind = case["kind"]
    blocks, thresh = _scene(case, seed)
    half = float(case["M"])
    scene = synth.Scene(blocks, (-half, -half, -1.0), (half, half, 1.0), thresh, OCC_CELL, OCC_THRESH)
    st = {"kind": kind, "case": case, "ctx": cow.Context(scene, case["storage"], bricks=case.get("bricks", False)),
          "mlp": _mlp(seed), "thresh": thresh, "ids": list(range(len(blocks)))}
    if kind in ("view", "batch", "optimise"):
        st["cams"] = [synth.Camera(*c) for c in _cameras(case, seed)]
    if kind == "view" and case["n_freq"] >= 0:
        st["ctx"].set_block_mlps(_block_mlps(seed, len(blocks), case["n_freq"]), case["n_freq"])
    if kind == "batch":
        st["batch"] = cow.Batch(st["ctx"], case["views"], case["views"] * len(blocks))
        n = sum(c.width * c.height for c in st["cams"])
        st["rgb"] = torch.empty((n, 3), device=DEV)
    if kind in ("eval", "autograd", "train", "train_block"):
        st["o"], st["d"], st["target"] = _rays(case, seed)
    if kind in ("autograd", "train", "train_block"):
        st["shapes"] = [p.shape for b in blocks for p in (b.grid, *b.planes)]
    if kind == "autograd":
        st["params"] = [p.requires_grad_() for b in blocks for p in (b.grid, *b.planes)]
        st["mlp"].requires_grad_()
    if kind == "train" and case["reg"]:
        st["points"] = _reg_points(case, seed)
    if kind == "train_block":
        st["block_mlps"] = _block_mlps(seed, len(blocks), case["n_freq"])
        st["ctx"].set_block_mlps(st["block_mlps"], case["n_freq"])
    if kind == "optimise":
        st["moments"] = _moments(case, seed, blocks)
        st["params"] = [p for b in blocks for p in (b.grid, *b.planes)]
        st["step"] = 100
    else:  # the context holds packed copies
        for b in blocks:
            b.grid, b.planes = None, []
    torch.cuda.empty_cache()
    return st


def _frame(st):
    """One frame of the viewer: LOD selection, then the render."""
    ctx, cam, ert = st["ctx"], st["cams"][0], st["case"].get("ert", 0.0)
    ids = ctx.select_lod(cam, st["thresh"])
    block_mlps = st["case"].get("n_freq", -1) >= 0
    return ctx.render([cam], [ids], None if block_mlps else st["mlp"], ert_eps=ert, block_mlps=block_mlps)[:2]


def _grad_tables(st):
    g = [torch.zeros(s, dtype=torch.float32, device=DEV) for s in st["shapes"]]
    nb = len(st["ids"])
    return g, [g[4 * i] for i in range(nb)], [g[4 * i + 1:4 * i + 4] for i in range(nb)]


def run(st):
    kind, case, ctx = st["kind"], st["case"], st["ctx"]
    if kind == "view":
        rgb, aux = _frame(st)
        return {"rgb": rgb, "aux": aux}
    if kind == "batch":
        ids = [ctx.select_lod(c, st["thresh"]) for c in st["cams"]]
        st["batch"].set_views(st["cams"], ids)
        st["batch"].render(st["mlp"], st["rgb"], ert_eps=case["ert"])
        return {"rgb": st["rgb"]}
    if kind == "eval":
        rgb, aux, _ = ctx.render_rays(st["o"], st["d"], st["ids"], st["mlp"], ert_eps=case["ert"])
        return {"rgb": rgb, "aux": aux}
    if kind == "autograd":
        rgb = train.render_rays(ctx, st["ids"], st["o"], st["d"], st["mlp"], st["params"])
        loss = torch.nn.functional.mse_loss(rgb, st["target"])
        grads = torch.autograd.grad(loss, [st["mlp"], *st["params"]])
        return {"rgb": rgb.detach(), "loss": loss.detach(), "mlp": grads[0], "features": list(grads[1:])}
    if kind == "train":
        o, d, ids, mlp = st["o"], st["d"], st["ids"], st["mlp"]
        block_T = None
        if case["reg"]:
            rgb, aux, block_T = ctx.render_rays_block_t(o, d, ids, mlp)
        else:
            rgb, aux, _ = ctx.render_rays(o, d, ids, mlp)
        g, loss = cow.mse_grad(rgb, st["target"])
        grads, gg, gp = _grad_tables(st)
        gm = torch.zeros_like(mlp)
        ctx.render_backward(o, d, ids, mlp, aux, g, gg, gp, gm)
        out = {"rgb": rgb, "loss": loss, "mlp": gm, "features": grads}
        if case["reg"]:
            reg = torch.zeros(1, dtype=torch.float32, device=DEV)
            ctx.sparsity_loss(st["points"], ids, REG_SPARSITY, loss=reg, grads=(gg, gp))
            ctx.opacity_loss(o, d, ids, REG_OPACITY, loss=reg, grads=(gg, gp), block_T=block_T)
            out["reg"] = reg
        return out
    if kind == "train_block":
        o, d, ids = st["o"], st["d"], st["ids"]
        rgb, state = ctx.render_rays_block_state(o, d, ids)
        g, loss = cow.mse_grad(rgb, st["target"])
        grads, gg, gp = _grad_tables(st)
        gm = torch.zeros_like(st["block_mlps"])
        ctx.render_backward_block_mlps_state(o, d, ids, state, g, gg, gp, gm)
        return {"rgb": rgb, "loss": loss, "mlp": gm, "features": grads}
    # optimise: Adam on every tensor, the render copies re-packed, a thumbnail of them
    st["step"] += 1
    for p, (g, m, v) in zip(st["params"], st["moments"]):
        cow.adam_step(p, g, m, v, 1e-2, st["step"])
    for i in st["ids"]:
        ctx.update_features(i, st["params"][4 * i], st["params"][4 * i + 1:4 * i + 4])
    rgb, aux = _frame(st)
    return {"params": list(st["params"]), "m": [m for _, m, _ in st["moments"]],
            "v": [v for _, _, v in st["moments"]], "rgb": rgb, "aux": aux}


# --------------------------------------------------------------------------
# what a pass cannot do without

SAMPLE_BYTES = {"fp32": 640, "fp16": 320, "bf16": 320, "fp8": 160, "bf16_fp8": 224, "fp8_bf16d": 176}
VERTEX_BYTES = {"fp32": (32, 32), "fp16": (16, 16), "bf16": (16, 16), "fp8": (8, 8), "bf16_fp8": (16, 8),
                "fp8_bf16d": (10, 8)}
LOOKUP_FLOPS, SHADE_FLOPS, MLP_FLOPS = 320, 100, 928


def work(case):
    """Features are counted once (or as the samples read them, where that is
    less), inputs and outputs once.  A camera ray meets opaque matter after
    about 0.4 units of occupied space, a ray without early termination passes
    about 1.5 (one block) or 2.1 of them; a unit holds P / 2 samples."""
    kind, n_blocks = case["kind"], case["M"] ** 2
    if case["levels"] > 1 and kind == "view":
        n_blocks /= 4  # the camera selects the near quarter at the finest level
    gb, pb = VERTEX_BYTES[case["storage"]]
    vertices, texels = n_blocks * case["R"] ** 3, n_blocks * 3 * case["P"] ** 2
    feat = vertices * gb + texels * pb
    params = 8 * (vertices + texels)
    if kind == "optimise":
        return {"bytes": params * 4 * 7 + feat, "flops": params * 12}
    if kind in ("view", "batch"):
        rays = (case["width"] * case["height"] if kind == "view" else case["views"] * 900000)
        samples = rays * 0.4 * case["P"] / 2
        out = rays * (44 if kind == "view" else 12)
        return {"bytes": min(feat, samples * SAMPLE_BYTES[case["storage"]]) + out,
                "flops": samples * (LOOKUP_FLOPS + SHADE_FLOPS) + rays * MLP_FLOPS}
    rays = case["n_rays"]
    samples = rays * (1.5 if case["M"] == 1 else 2.1) * case["P"] / 2
    read = min(feat, samples * SAMPLE_BYTES[case["storage"]])
    if kind == "eval":
        return {"bytes": read + rays * (24 + 44), "flops": samples * (LOOKUP_FLOPS + SHADE_FLOPS) + rays * MLP_FLOPS}
    return {"bytes": read + params * 4 + rays * 48,
            "flops": samples * (2 * (LOOKUP_FLOPS + SHADE_FLOPS) + LOOKUP_FLOPS) + rays * 3 * MLP_FLOPS}


# --------------------------------------------------------------------------
# the same in 64 bits


def _fp8(x):
    """E4M3 with the smallest power-of-two scale per channel that fits."""
    top = x.reshape(-1, 8).abs().amax(0).double() / 448.0
    m, e = torch.frexp(top)
    s = torch.where(top > 0, torch.ldexp(torch.ones_like(m), torch.where(m == 0.5, e - 1, e)), torch.ones_like(m))
    s = s.float()
    return (x / s).to(torch.float8_e4m3fn).float() * s


def _stored(x, storage, grid):
    if storage == "fp32":
        return x
    if storage == "fp16":
        return x.half().float()
    if storage == "bf16" or (storage == "bf16_fp8" and grid):
        return x.bfloat16().float()
    y = _fp8(x)
    if storage == "fp8_bf16d" and grid:
        y[..., 0] = x[..., 0].bfloat16().float()
    return y


class _Exact:
    """One block in 64 bits: its occupancy from the master, its features as stored."""

    def __init__(self, b, storage):
        self.lo, self.hi, self.R, self.P, self.level, self.parent = b.lo, b.hi, b.R, b.P, b.level, b.parent
        nc = -(-(b.R - 1) // OCC_CELL)
        pad = nc * OCC_CELL + 1 - b.R
        th = math.log(float(np.float32(OCC_THRESH)))
        occ = (b.grid[..., 0].double() > th).float()
        occ = torch.nn.functional.pad(occ, (0, pad, 0, pad, 0, pad))
        self.occ = torch.nn.functional.max_pool3d(occ[None, None], OCC_CELL + 1, OCC_CELL)[0, 0] > 0
        rows = torch.nonzero(self.occ.any(2).any(1)).flatten()
        top = min((int(rows[-1]) + 1) * OCC_CELL, b.R - 1) if len(rows) else 0
        self.ztop = self.lo[2] + top * (self.hi[2] - self.lo[2]) / (b.R - 1)
        self.master, self.storage, self.feat = [b.grid, *b.planes], storage, None

    def load(self):
        if self.feat is None:
            self.feat = [_stored(x, self.storage, k == 0).reshape(-1, 8) for k, x in enumerate(self.master)]
        return self

    def unload(self):
        self.feat = None

    def samples(self, o, d, most=3 << 20):
        """The occupied lattice samples of FP32 rays, in chunks of whole rays:
        (first ray, last ray, ray of each sample, sample index)."""
        delta = float(np.float32((self.hi[0] - self.lo[0]) / self.P))
        dl = torch.tensor(delta, dtype=torch.float32, device=DEV)
        o64, d64 = o.double(), d.double()
        lo, hi = (torch.tensor(v, dtype=torch.float64, device=DEV) for v in (self.lo, self.hi))
        t0, t1 = (lo - 1e-2 - o64) / d64, (hi + 1e-2 - o64) / d64
        tn = torch.minimum(t0, t1).nan_to_num(-1e30, 1e30, -1e30).amax(1).clamp(min=0)
        tf = torch.maximum(t0, t1).nan_to_num(1e30, 1e30, -1e30).amin(1)
        i0 = (torch.floor(tn / delta) - 3).clamp(min=0).long()
        n = torch.where(tf >= tn, torch.ceil(tf / delta).clamp(max=1e9).long() + 3 - i0, 0).clamp(min=0)
        ends = torch.cumsum(n, 0).cpu().numpy()
        a = 0
        lof, hif = lo.float(), hi.float()
        kg = torch.tensor([(self.R - 1) / (self.hi[k] - self.lo[k]) for k in range(3)], dtype=torch.float64,
                          device=DEV).float()
        while a < len(ends):
            base = int(ends[a - 1]) if a else 0
            b = max(a + 1, int(np.searchsorted(ends, base + most, side="right")))
            if int(ends[b - 1]) > base:
                ray = torch.repeat_interleave(torch.arange(a, b, device=DEV), n[a:b])
                first = torch.cumsum(n[a:b], 0) - n[a:b]
                i = torch.arange(len(ray), device=DEV) - first[ray - a] + i0[ray]
                t = (i.float() + 0.5) * dl
                p = d[ray] * t[:, None]
                p = p + o[ray]
                ok = (p >= lof).all(1) & (p[:, :2] < hif[:2]).all(1) & (p[:, 2] <= hif[2])
                ray, i, p = ray[ok], i[ok], p[ok]
                g = p - lof
                g = g * kg
                cell = torch.floor(g).clamp(0, self.R - 2).long() // OCC_CELL
                ok = self.occ[cell[:, 2], cell[:, 1], cell[:, 0]]
                yield a, b, ray[ok], i[ok]
            a = b
        return

    def points(self, o, d, ray, i):
        delta = float(np.float32((self.hi[0] - self.lo[0]) / self.P))
        return o[ray].double() + ((i.double() + 0.5) * delta)[:, None] * d[ray].double()

    def taps(self, p):
        """(tensor, vertex index, weight) of the 8 + 12 taps at points p."""
        lo, hi = (torch.tensor(v, dtype=torch.float64, device=DEV) for v in (self.lo, self.hi))
        out = []
        for n, tensors in ((self.R, (0,)), (self.P, (1, 2, 3))):
            g = ((p - lo) * ((n - 1) / (hi - lo))).clamp(0, n - 1)
            c = torch.floor(g).clamp(0, n - 2)
            f, c = g - c, c.long()
            for t in tensors:
                axes = ((0, 1, 2), (0, 1), (0, 2), (1, 2))[t]
                for k in range(1 << len(axes)):
                    idx, w = 0, 1.0
                    for q, ax in enumerate(axes):
                        bit = (k >> q) & 1
                        idx = idx + (c[:, ax] + bit) * n ** q
                        w = w * (f[:, ax] if bit else 1 - f[:, ax])
                    out.append((t, idx, w))
        return out

    def lookup(self, taps):
        f = torch.zeros((len(taps[0][1]), 8), dtype=torch.float64, device=DEV)
        for t, idx, w in taps:
            f.addcmul_(self.feat[t][idx].double(), w[:, None])
        return f

    def march(self, o, d, B=None, ert=0.0, up=None, grads=None):
        """(C^k, F^k, T^k, whether the ray has a sample); with up = (dL/dC^k,
        dL/dF^k, dL/dT^k) the feature gradients go to `grads` instead."""
        self.load()
        delta = float(np.float32((self.hi[0] - self.lo[0]) / self.P))
        N = len(o)
        CF = torch.zeros((N, 7), dtype=torch.float64, device=DEV)
        tau_ray = torch.zeros(N, dtype=torch.float64, device=DEV)
        has = torch.zeros(N, dtype=torch.bool, device=DEV)
        for _, _, ray, i in self.samples(o, d):
            if not len(ray):
                continue
            taps = self.taps(self.points(o, d, ray, i))
            f = self.lookup(taps)
            tau = torch.exp(f[:, 0]) * delta
            start = torch.ones_like(ray, dtype=torch.bool)
            start[1:] = ray[1:] != ray[:-1]
            seg = torch.cumsum(start, 0) - 1

            def before(x):  # sum of a ray's earlier samples
                c = torch.cumsum(x, 0) - x
                return c - c[start][seg]

            T = torch.exp(-before(tau))
            if ert > 0.0:
                keep = T * (1.0 if B is None else B[ray]) >= ert
            else:
                keep = torch.ones_like(start)
            w = torch.where(keep, T * -torch.expm1(-tau), 0.0)
            c = torch.sigmoid(f[:, 1:])
            if up is None:
                CF.index_add_(0, ray, w[:, None] * c)
                tau_ray.index_add_(0, ray, torch.where(keep, tau, 0.0))
                has[ray[keep]] = True
                continue
            gCF, gT = up
            dot = (gCF[ray] * c).sum(1)
            total = torch.zeros(int(seg[-1]) + 1, dtype=torch.float64, device=DEV).index_add_(0, seg, w * dot)
            tail = torch.zeros_like(total).index_add_(0, seg, tau)
            later = total[seg] - before(w * dot) - w * dot
            g = torch.empty_like(f)
            g[:, 0] = tau * (T * torch.exp(-tau) * dot - later - gT[ray] * torch.exp(-tail)[seg])
            g[:, 1:] = w[:, None] * gCF[ray] * c * (1 - c)
            for t, idx, tw in taps:
                grads[t].index_add_(0, idx, tw[:, None] * g)
        self.unload()
        return CF, torch.exp(-tau_ray), has


def _shade(mlp, n_in, x):
    """The deferred MLP n_in -> 16 -> 16 -> 3 of parameters mlp, sigmoid output."""
    k = 16 * n_in
    W1, b1 = mlp[:k].view(n_in, 16), mlp[k:k + 16]
    W2, b2 = mlp[k + 16:k + 272].view(16, 16), mlp[k + 272:k + 288]
    W3, b3 = mlp[k + 288:k + 336].view(16, 3), mlp[k + 336:k + 339]
    h = torch.relu(torch.relu(x @ W1 + b1) @ W2 + b2)
    return torch.sigmoid(h @ W3 + b3)


def _encode(d, n_freq):
    out = [d]
    for k in range(n_freq):
        out += [torch.sin(2.0 ** k * d), torch.cos(2.0 ** k * d)]
    return torch.cat(out, 1)


def _pixel_rays(cam):
    """FP32 rays through the pixel centres, one IEEE operation at a time."""
    c2w, W, H, fov = cam
    f32 = dict(dtype=torch.float32, device=DEV)
    n = W * H
    full = lambda v: torch.full((n,), float(np.float32(v)), **f32)  # noqa: E731
    i = torch.arange(n, device=DEV)
    f = full((0.5 * H) / math.tan(0.5 * fov * math.pi / 180.0))
    xc = ((i % W).float() + 0.5 - full(0.5) * full(W)) / f
    yc = -(((i // W).float() + 0.5 - full(0.5) * full(H)) / f)
    dw = [(full(c2w[r][0]) * xc + full(c2w[r][1]) * yc) - full(c2w[r][2]) for r in range(3)]
    norm = torch.sqrt((dw[0] * dw[0] + dw[1] * dw[1]) + dw[2] * dw[2])
    return (torch.stack([full(c2w[r][3]) for r in range(3)], 1), torch.stack([v / norm for v in dw], 1))


def _select(blocks, cam, thresh):
    """LOD choice and depth order of one camera."""
    c2w, W, H, fov = cam
    m, t = np.asarray(c2w)[:, :3], np.asarray(c2w)[:, 3]
    f = (0.5 * H) / math.tan(0.5 * fov * math.pi / 180.0)
    kx, ky = W / (2 * f), H / (2 * f)

    def visible(b):
        q = np.array([[(b.hi if k & 1 else b.lo)[0], (b.hi if k & 2 else b.lo)[1],
                       b.ztop if k & 4 else b.lo[2]] for k in range(8)]) - t
        x, y, z = (q @ m).T
        z = -z
        return not any((s < 0).all() for s in (z, x + kx * z, kx * z - x, y + ky * z, ky * z - y))

    def distance(b):
        return math.hypot(0.5 * (b.lo[0] + b.hi[0]) - t[0], 0.5 * (b.lo[1] + b.hi[1]) - t[1], b.ztop - t[2])

    top = max(b.level for b in blocks)
    todo, out = [i for i, b in enumerate(blocks) if b.level == top and visible(b)], []
    while todo:
        i = todo.pop()
        kids = [k for k, b in enumerate(blocks) if b.parent == i and visible(b)]
        if blocks[i].level == 1 or all(distance(blocks[k]) > thresh[blocks[k].level - 1] for k in kids):
            out.append(i)
        else:
            todo += kids
    return sorted(out, key=lambda i: ((0.5 * (blocks[i].lo[0] + blocks[i].hi[0]) - t[0]) ** 2
                                      + (0.5 * (blocks[i].lo[1] + blocks[i].hi[1]) - t[1]) ** 2, i))


def _exact_view(blocks, cam, thresh, ert, mlp, block_mlps=None, n_freq=0):
    o, d = _pixel_rays(cam)
    N = len(o)
    CF = torch.zeros((N, 7), dtype=torch.float64, device=DEV)
    rgb = torch.zeros((N, 3), dtype=torch.float64, device=DEV)
    T = torch.ones(N, dtype=torch.float64, device=DEV)
    ert = float(np.float32(ert))
    enc = _encode(d.double(), n_freq if block_mlps is not None else 0)
    for i in _select(blocks, cam, thresh):
        cf, Tk, has = blocks[i].march(o, d, T, ert)
        if block_mlps is not None:
            phi = _shade(block_mlps[i].double(), enc.shape[1] + 7, torch.cat([cf, enc], 1))
            rgb += torch.where(has[:, None], T[:, None] * (cf[:, :3] + phi), 0.0)
        CF += T[:, None] * cf
        T = T * Tk
    if block_mlps is None:
        rgb = CF[:, :3] + _shade(mlp.double(), 10, torch.cat([CF, enc], 1))
    return rgb, torch.cat([CF, T[:, None]], 1)


def _ray_order(blocks, o):
    """Per ray the blocks by the xy distance of their centres, FP32 keys, ties by index."""
    keys = []
    for b in blocks:
        c = [float(np.float32((b.lo[k] + b.hi[k]) / 2)) for k in range(2)]
        dx, dy = (torch.full_like(o[:, k], c[k]) - o[:, k] for k in range(2))
        keys.append(dx * dx + dy * dy)
    return torch.sort(torch.stack(keys, 1), dim=1, stable=True)[1]


def _over(order, CF, Tk, has=None):
    """Blocks in each ray's order: (C_d and F weights, transmittance in front, order-gathered)."""
    T = torch.gather(Tk, 1, order)
    B = torch.cumprod(torch.cat([torch.ones_like(T[:, :1]), T], 1), 1)
    cf = torch.gather(CF, 1, order[..., None].expand(-1, -1, 7))
    return cf, B


def exact(case, seed):
    kind = case["kind"]
    masters, thresh = _scene(case, seed)
    mlp = _mlp(seed)
    if kind == "optimise":
        return _exact_optimise(case, seed, masters, thresh, mlp)
    blocks = [_Exact(b, case["storage"]) for b in masters]
    if kind == "view":
        bm = _block_mlps(seed, len(blocks), case["n_freq"]) if case["n_freq"] >= 0 else None
        rgb, aux = _exact_view(blocks, _cameras(case, seed)[0], thresh, case["ert"], mlp, bm, max(case["n_freq"], 0))
        return {"rgb": rgb, "aux": aux}
    if kind == "batch":
        return {"rgb": torch.cat([_exact_view(blocks, c, thresh, case["ert"], mlp)[0]
                                  for c in _cameras(case, seed)])}
    o, d, target = _rays(case, seed)
    order = _ray_order(blocks, o)
    if kind == "eval":
        return _exact_eval(case, blocks, o, d, order, mlp)
    return _exact_train(case, seed, blocks, o, d, target, order, mlp)


def _exact_optimise(case, seed, masters, thresh, mlp):
    out = {"params": [], "m": [], "v": []}
    blocks = [_Exact(b, case["storage"]) for b in masters]
    step, moments = 101, _moments(case, seed, masters)
    bc1, bc2 = 1 - 0.9 ** step, 1 - 0.999 ** step
    for b, x in zip(masters, blocks):
        for k, p in enumerate((b.grid, *b.planes)):
            g, m, v = (t.double() for t in moments.pop(0))
            m = 0.9 * m + (1 - 0.9) * g
            v = 0.999 * v + (1 - 0.999) * g * g
            q = p.double() - 1e-2 * (m / bc1) / (torch.sqrt(v / bc2) + 1e-8)
            x.master[k] = q.float()
            out["params"].append(q)
            out["m"].append(m)
            out["v"].append(v)
    out["rgb"], out["aux"] = _exact_view(blocks, _cameras(case, seed)[0], thresh, 0.0, mlp)
    return out


def _exact_eval(case, blocks, o, d, order, mlp):
    N, nb = len(o), len(blocks)
    ert = float(np.float32(case["ert"]))
    CF, Tk = _partials(blocks, o, d)
    if ert > 0.0:  # again, each block's samples up to the ray's termination
        _, B = _over(order, CF, Tk)
        front = torch.empty((N, nb), dtype=torch.float64, device=DEV).scatter_(1, order, B[:, :-1])
        CF, Tk = _partials(blocks, o, d, front, ert)
    cf, B = _over(order, CF, Tk)
    cf = (B[:, :-1, None] * cf).sum(1)
    rgb = cf[:, :3] + _shade(mlp.double(), 10, torch.cat([cf, d.double()], 1))
    return {"rgb": rgb, "aux": torch.cat([cf, B[:, -1:]], 1)}


def _partials(blocks, o, d, front=None, ert=0.0):
    got = [b.march(o, d, None if front is None else front[:, k], ert) for k, b in enumerate(blocks)]
    return torch.stack([g[0] for g in got], 1), torch.stack([g[1] for g in got], 1)


def _exact_train(case, seed, blocks, o, d, target, order, mlp):
    got = [b.march(o, d) for b in blocks]
    CF = torch.stack([g[0] for g in got], 1).requires_grad_()
    Tk = torch.stack([g[1] for g in got], 1).requires_grad_()
    cf, B = _over(order, CF, Tk)
    d64 = d.double()
    if case["kind"] == "train_block":
        w = _block_mlps(seed, len(blocks), case["n_freq"]).double().requires_grad_()
        enc = _encode(d64, case["n_freq"])
        front = torch.zeros_like(Tk).scatter(1, order, B[:, :-1])
        rgb = 0.0
        for k in range(len(blocks)):
            x = CF[:, k, :3] + _shade(w[k], enc.shape[1] + 7, torch.cat([CF[:, k], enc], 1))
            rgb = rgb + torch.where(got[k][2][:, None], front[:, k:k + 1] * x, 0.0)
    else:
        w = mlp.detach().double().requires_grad_()
        cf = (B[:, :-1, None] * cf).sum(1)
        rgb = cf[:, :3] + _shade(w, 10, torch.cat([cf, d64], 1))
    loss = ((rgb - target.double()) ** 2).mean()
    total, reg = loss, None
    if case.get("reg"):
        has = torch.stack([g[2] for g in got], 1)
        a = (1 - Tk).clamp(1e-6, 1 - 1e-6)
        ent = torch.where(has, -(a * torch.log(a) + (1 - a) * torch.log1p(-a)), 0.0).sum() / len(o)
        reg = REG_OPACITY * ent
        total = loss + reg
    gw, gCF, gT = torch.autograd.grad(total, [w, CF, Tk])
    feats = []
    for k, b in enumerate(blocks):
        grads = [torch.zeros((n, 8), dtype=torch.float64, device=DEV) for n in [b.R ** 3] + [b.P ** 2] * 3]
        b.march(o, d, up=(gCF[:, k], gT[:, k]), grads=grads)
        if case.get("reg"):
            reg = reg + _exact_sparsity(case, seed, b, grads)
        feats += [g.view(*([b.R] * 3 if t == 0 else [b.P] * 2), 8) for t, g in enumerate(grads)]
    out = {"rgb": rgb.detach(), "loss": loss.detach(), "mlp": gw, "features": feats}
    if case["kind"] != "autograd":
        out["loss"] = out["loss"].view(1)
    if case.get("reg"):
        out["reg"] = reg.detach().view(1)
    return out


def _exact_sparsity(case, seed, b, grads):
    p = _reg_points(case, seed)
    lo, hi = (torch.tensor(v, dtype=torch.float32, device=DEV) for v in (b.lo, b.hi))
    p = p[(p >= lo).all(1) & (p[:, :2] < hi[:2]).all(1) & (p[:, 2] <= hi[2])].double()
    delta = float(np.float32((b.hi[0] - b.lo[0]) / b.P))
    b.load()
    taps = b.taps(p)
    tau = torch.exp(b.lookup(taps)[:, 0]) * delta
    b.unload()
    scale = REG_SPARSITY / REG_POINTS
    for t, idx, w in taps:
        grads[t][:, 0].index_add_(0, idx, w * scale * tau * torch.exp(-tau))
    return scale * -torch.expm1(-tau).sum()
