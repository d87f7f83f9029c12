"""Performance cases of the Fourier PlenOctree renderer.

Each case is one call (or one training step) that a program using this package
makes, through the package's public entry points:

  frame     Renderer.render of one camera frame, single call, waited for or not:
            an interactive viewer.
  frames    Renderer.render_frames of several frames: video export, free-viewpoint
            playback (every frame has its own time) or several views of one time.
  rays      render_rays and its backward on explicit rays with per-ray times: a
            differentiable render inside a program's own loss.
  finetune  FineTuner.step: forward, squared error, adjoint and sparse Adam.
  dft       dft_leaves: per-frame leaf values to Fourier coefficients, the
            generation of a Fourier PlenOctree.
  latent    LatentModel.step: one optimiser step of the latent decoder.
  pixel     PixelLoss.gradient: decode of every leaf, two renders and the adjoint,
            the rendered-pixel term of the decoder's training.

Trees are the animated capsule body of `synth` (the union over `body_frames`
frames on a 2^depth grid) or the spherical shell of the parity workload.
`exact` evaluates the same quantities in plain torch FP64, with a cell-by-cell
walk of a dense grid in place of the octree.
"""

import functools
import math

import numpy as np
import torch

from paper_2202_08614_gb300 import fpo, synth
from paper_2202_08614_gb300.finetune import FineTuner, camera_ray_batch
from paper_2202_08614_gb300.latent import LatentModel, PixelLoss

DEV = "cuda"
PERIOD = synth.PERIOD_T
BG, STOP_T = (1.0, 1.0, 1.0), 1e-4
LR, BETAS, EPS = 1e-2, (0.9, 0.999), 1e-8
FIT_STEPS = 400  # optimiser steps that a training state has behind it

BODY = {"tree": "body", "n1": 31, "n2": 5}


def listed():
    return [
        # a preview: the 128x128 frame of a 5,096-leaf tree; launches and latency are all there is
        {"name": "frame_shell_128", "kind": "frame", "tree": "shell", "depth": 5, "body_frames": 1, "n1": 31, "n2": 5,
         "storage": "f32", "width": 128, "height": 128},
        # one full-HD frame of the 512^3 body on request (a viewer that reacts to its user)
        {"name": "frame_f32_1080p", "kind": "frame", **BODY, "depth": 9, "body_frames": 60, "storage": "f32",
         "width": 1920, "height": 1080},
        # playback: eight full-HD frames, each at its own time
        {"name": "frames_f32_1080p", "kind": "frames", **BODY, "depth": 9, "body_frames": 60, "storage": "f32",
         "width": 1920, "height": 1080, "count": 8, "one_t": False},
        # playback from half-size BF16 coefficients in an odd window
        {"name": "frames_bf16_odd", "kind": "frames", **BODY, "depth": 8, "body_frames": 20, "storage": "bf16",
         "width": 1001, "height": 563, "count": 5, "one_t": False},
        # playback of a compressed scene (per-leaf latents and the shared decoder), 800x800
        {"name": "frames_latent_800", "kind": "frames", **BODY, "depth": 8, "body_frames": 60, "storage": "latent",
         "width": 800, "height": 800, "count": 6, "one_t": False},
        # several views of one moment from FP8 coefficients (a light-field display)
        {"name": "views_fp8_540p", "kind": "frames", **BODY, "depth": 7, "body_frames": 60, "storage": "fp8",
         "width": 960, "height": 540, "count": 5, "one_t": True},
        # a differentiable render of a small ray batch in a user's own training loop
        {"name": "rays_grad_4095", "kind": "rays", **BODY, "depth": 7, "body_frames": 60, "rays": 4095},
        # fine-tuning of the full body: 65,536 rays over 16 views x 60 frames at 800x800
        {"name": "finetune_65536", "kind": "finetune", **BODY, "depth": 9, "body_frames": 60, "rays": 65536},
        # generation: Fourier coefficients of a chunk of leaves from 60 frames
        {"name": "dft_262147", "kind": "dft", "leaves": 262147, "frames": 60, "n1": 31, "n2": 5},
        # a training step of the latent decoder on the tensor cores
        {"name": "latent_step_tc_65536", "kind": "latent", "leaves": 600000, "batch": 65536, "n1": 31, "n2": 5,
         "tensor_cores": True},
        # the same in FP32 on a small odd batch
        {"name": "latent_step_fp32_8191", "kind": "latent", "leaves": 100003, "batch": 8191, "n1": 31, "n2": 5,
         "tensor_cores": False},
        # the rendered-pixel term of the decoder's training
        {"name": "pixel_loss_8192", "kind": "pixel", **BODY, "depth": 8, "body_frames": 60, "rays": 8192,
         "tensor_cores": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frames", "frames", "rays", "finetune", "dft", "latent", "pixel"])
    n1, n2 = rng.choice([(31, 5), (31, 5), (21, 5), (11, 5), (31, 11)])
    body = {"tree": "body", "n1": n1, "n2": n2, "depth": rng.choice([6, 7, 8]), "body_frames": _log_int(rng, 1, 60)}
    if kind in ("frame", "frames"):
        storage = rng.choice(["f32", "f32", "bf16", "f16", "fp8", "latent"])
        if storage in ("bf16", "f16", "fp8"):
            body["depth"] = min(body["depth"], 7)
        elif storage == "latent" and n1 + 27 * n2 > 176:
            body["n2"] = 5
        c = {"kind": kind, **body, "storage": storage, "width": _log_int(rng, 96, 1920), "height": _log_int(rng, 96, 1080)}
        if kind == "frames":
            c.update(count=rng.randint(2, 7), one_t=rng.random() < 0.25)
        return c
    if kind in ("rays", "finetune"):
        return {"kind": kind, **body, "rays": _log_int(rng, 1000, 65536)}
    if kind == "dft":
        return {"kind": kind, "leaves": _log_int(rng, 2000, 262147), "frames": rng.choice([24, 60, 60, 75, 100]), "n1": n1,
                "n2": n2}
    tc = rng.random() < 0.6
    if kind == "latent":
        batch = _log_int(rng, 2000, 65536)
        return {"kind": kind, "leaves": batch + _log_int(rng, 10000, 500000), "batch": batch, "n1": n1, "n2": 5,
                "tensor_cores": tc}
    return {"kind": kind, **body, "n2": 5, "rays": _log_int(rng, 2000, 16384), "tensor_cores": tc}


# --------------------------------------------------------------------------
# inputs


@functools.lru_cache(maxsize=4)
def _cells(tree, depth, body_frames):
    """Leaf cells uint32 [n, 3] in Morton order (host)."""
    if tree == "shell":
        return synth.shell_leaves(depth)
    a, b, r = synth.capsule_body(np.random.default_rng(0), n_frames=body_frames)
    dev = lambda x: torch.as_tensor(x, dtype=torch.float32, device=DEV)
    A, B = dev(a).reshape(-1, 3), dev(b).reshape(-1, 3)
    R = dev(r)[:, None].expand(len(r), body_frames).reshape(-1)
    ab = B - A
    ab2 = (ab * ab).sum(1)
    oct_ = torch.tensor([[k & 1, (k >> 1) & 1, (k >> 2) & 1] for k in range(8)], device=DEV)
    cand = torch.zeros((1, 3), dtype=torch.int64, device=DEV)
    for level in range(1, depth + 1):
        cand = (cand[:, None] * 2 + oct_).reshape(-1, 3)
        h = 1.0 / (1 << level)
        span = 0.5 * math.sqrt(3.0) * (h - 1.0 / (1 << depth))  # centre to the farthest finest-cell centre
        keep = []
        step = max(1, (1 << 26) // A.shape[0])
        for s in range(0, cand.shape[0], step):
            ctr = (cand[s:s + step].float() + 0.5) * h
            ap = ctr[:, None] - A[None]
            t = ((ap * ab).sum(-1) / ab2).clamp(0.0, 1.0)
            dist = (ap - t[..., None] * ab).norm(dim=-1)
            keep.append((dist - span <= R).any(1))
        cand = cand[torch.cat(keep)]
    return cand.to(torch.int32).cpu().numpy().astype(np.uint32)


def _case_cells(case):
    return _cells(case["tree"], case["depth"], case["body_frames"])


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFF)


def _coef_std(n1, n2):
    """Standard deviation of each canonical coefficient (the mean is 0; k_sigma_0 ~ U(0, 50))."""
    sig = 5.0 / (torch.arange(n1, device=DEV) + 1.0)
    z = 0.2 / (torch.arange(n2, device=DEV) + 1.0)
    z[0] = 0.5
    return torch.cat([sig, z.repeat(27)])


def _coeffs(gen, n, n1, n2):
    """Coefficients [n, n1 + 27 n2] with the distributions of synth.draw_coefficients, drawn on the GPU."""
    c = torch.empty((n, n1 + 27 * n2), device=DEV).normal_(generator=gen)
    c *= _coef_std(n1, n2)
    c[:, 0] = torch.rand(n, generator=gen, device=DEV) * 50.0
    return c


def _tree(case, coeffs):
    """The tree that Renderer.upload takes; `coeffs` is a host array."""
    xyz = _case_cells(case)
    return synth.Tree(np.full(xyz.shape[0], case["depth"], np.uint8), xyz, coeffs, case["depth"], case["n1"], case["n2"])


def _renderer(case, coeffs, **kw):
    """A renderer with the tree uploaded and FP32 coefficients set from the GPU array `coeffs`."""
    r = fpo.Renderer(n1=case["n1"], n2=case["n2"], period_T=PERIOD, **kw)
    r.upload(_tree(case, np.zeros(tuple(coeffs.shape), np.float32)))
    r.set_coeffs(coeffs)
    return r


def _views(case, seed):
    rng = np.random.default_rng(seed)
    count = case.get("count", 1)
    cams = [synth.Camera(eye=synth.sphere_eye(float(rng.uniform(0, 360)), float(rng.uniform(-10, 30))),
                         width=case["width"], height=case["height"]) for _ in range(count)]
    times = [float(rng.integers(0, 60)) for _ in range(count)]
    if case.get("one_t"):
        times = times[:1] * count
    elif case["tree"] == "shell":
        times = [float(rng.uniform(0, 60))]
    return cams, times


def _decoder(gen, n, n1, n2):
    """Latents and decoder weights whose outputs are spread like the coefficients above."""
    rn = lambda *s: torch.randn(*s, generator=gen, device=DEV)
    w = {"lat": rn(n, 32) * 0.5, "w1": rn(64, 32) * math.sqrt(2 / 32), "b1": rn(64) * 0.1,
         "w2": rn(64, 64) * math.sqrt(2 / 64), "b2": rn(64) * 0.1}
    std = _coef_std(n1, n2)
    std[0] = 12.0
    w["w3"] = rn(n1 + 27 * n2, 64) * (std / 4.0)[:, None]
    w["b3"] = rn(n1 + 27 * n2) * std * 0.2
    w["b3"][0] = 25.0
    return w


def _ring():
    return synth.ring_cameras(16, 800, 800)


def _batch(case, gen):
    """Training rays over 16 views and 60 frames, and a smooth picture as their target colours."""
    o, d, t = camera_ray_batch(_ring(), case["rays"], gen)
    f = torch.tensor([[3.0, 1.0, 2.0], [1.0, 4.0, -2.0], [-2.0, 2.0, 3.0]], device=DEV)
    y = 0.5 + 0.4 * torch.sin(d @ f.T + o @ f + t[:, None] * (2 * math.pi / PERIOD))
    return o, d, t, y.contiguous()


def _moments(gen, shape, scale):
    """Adam moments of a run under way: gradients of about `scale`."""
    m = torch.randn(shape, generator=gen, device=DEV) * (0.3 * scale)
    v = (torch.rand(shape, generator=gen, device=DEV) + 0.5) * (scale * scale)
    return m, v


def _latent_inputs(case, seed):
    g = _gen(seed)
    n, nc = case["leaves"], case["n1"] + 27 * case["n2"]
    w = _decoder(g, n, case["n1"], case["n2"])
    mv = {k: _moments(g, x.shape, 1e-4 if k == "lat" else 1e-2) for k, x in w.items()}
    targets = _coeffs(g, n, case["n1"], case["n2"])
    rows = torch.randperm(n, generator=g, device=DEV)[: case["batch"]].to(torch.int32)
    cw = torch.ones(nc, device=DEV)
    cw[: case["n1"]] = 0.05
    return w, mv, targets, rows, cw / nc


def _dft_values(case, seed):
    """Per-frame leaf values: a clipped density and travelling waves of colour."""
    g = _gen(seed)
    T, n = case["frames"], case["leaves"]
    t = torch.arange(1, T + 1, device=DEV)[:, None, None] * (2 * math.pi / T)
    a = torch.randn((3, n, 28), generator=g, device=DEV)
    v = a[0] + a[1] * torch.sin(t + a[2])
    v[..., 0] = v[..., 0].clamp_min(0.0) * 20.0
    return v


def _fine_inputs(case, seed):
    g = _gen(seed)
    n = _case_cells(case).shape[0]
    c = _coeffs(g, n, case["n1"], case["n2"])
    return c, _batch(case, g), _moments(g, c.shape, 1e-6), g


# --------------------------------------------------------------------------
# the cases


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind in ("frame", "frames"):
        g = _gen(seed)
        n = _case_cells(case).shape[0]
        s["cams"], s["times"] = _views(case, seed)
        if case["storage"] == "latent":
            s["r"] = fpo.Renderer(n1=case["n1"], n2=case["n2"], period_T=PERIOD, storage="latent")
            s["r"].upload(_tree(case, np.zeros(1, np.float32)))
            w = _decoder(g, n, case["n1"], case["n2"])
            s["r"].set_latents(w["lat"].half(), *(w[k] for k in ("w1", "b1", "w2", "b2", "w3", "b3")))
        elif case["storage"] == "f32":
            s["r"] = _renderer(case, _coeffs(g, n, case["n1"], case["n2"]))
        else:
            s["r"] = fpo.Renderer(n1=case["n1"], n2=case["n2"], period_T=PERIOD, storage=case["storage"])
            s["r"].upload(_tree(case, _coeffs(g, n, case["n1"], case["n2"]).cpu().numpy()))
    elif kind == "rays":
        s["coeffs"], s["batch"], _, _ = _fine_inputs(case, seed)
        s["r"] = _renderer(case, s["coeffs"])
    elif kind == "finetune":
        c, s["batch"], (m, v), _ = _fine_inputs(case, seed)
        s["r"] = _renderer(case, c)
        s["tuner"] = FineTuner(s["r"], c, lr=LR, betas=BETAS, eps=EPS, bg=BG, stop_T=STOP_T)
        s["tuner"].m.copy_(m)
        s["tuner"].v.copy_(v)
        s["tuner"].steps = FIT_STEPS
    elif kind == "dft":
        s["values"] = _dft_values(case, seed)
        s["sizes"] = {"n1": case["n1"], "n2": case["n2"]}
        s["out"] = torch.empty((case["leaves"], case["n1"] + 27 * case["n2"]), device=DEV)
        s["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    elif kind == "latent":
        w, mv, s["targets"], s["rows"], s["cw"] = _latent_inputs(case, seed)
        s["model"] = LatentModel(case["leaves"], case["n1"], case["n2"], tensor_cores=case["tensor_cores"])
        for k, x in w.items():
            s["model"].p[k].copy_(x)
            s["model"].m[k].copy_(mv[k][0])
            s["model"].v[k].copy_(mv[k][1])
        s["model"].step_count = FIT_STEPS
    else:
        g = _gen(seed)
        n = _case_cells(case).shape[0]
        w = _decoder(g, n, case["n1"], case["n2"])
        s["model"] = LatentModel(n, case["n1"], case["n2"], tensor_cores=case["tensor_cores"])
        for k, x in w.items():
            s["model"].p[k].copy_(x)
        coeffs = _coeffs(g, n, case["n1"], case["n2"]).cpu().numpy()
        s["loss"] = PixelLoss(_tree(case, coeffs), _ring(), rays=case["rays"], weight=10.0, seed=int(seed) & 0x7FFFFFFF,
                              bg=BG, stop_T=STOP_T, tensor_cores=case["tensor_cores"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "frame":
        return s["r"].render(camera=s["cams"][0], t=s["times"][0], bg=BG, stop_T=STOP_T)["rgb"]
    if kind == "frames":
        return s["r"].render_frames(s["cams"], s["times"], bg=BG, stop_T=STOP_T)
    if kind == "rays":
        o, d, t, y = s["batch"]
        c = s["coeffs"].detach().requires_grad_()
        rgb = fpo.render_rays(c, s["r"], o, d, t, BG, STOP_T)
        ((rgb - y) ** 2).sum(1).mean().backward()
        return {"rgb": rgb.detach(), "grad": c.grad}
    if kind == "finetune":
        tn = s["tuner"]
        loss = tn.step(*s["batch"])
        return {"loss": loss, "param": tn.param, "m": tn.m, "v": tn.v}
    if kind == "dft":
        return fpo.dft_leaves(s["values"], out=s["out"], status=s["status"], **s["sizes"])
    if kind == "latent":
        md = s["model"]
        loss = md.step(s["rows"], s["targets"], s["cw"])
        return {"loss": loss, "p": md.p, "m": md.m, "v": md.v, "g": md.g}
    _, dy = s["loss"].gradient(s["model"])
    return {"loss": s["loss"].last_loss, "dy": dy, "mark": s["loss"].mark}


VISITS = 9  # leaf segments of an average ray over the whole picture (18.1M visits per 1920x1080 body frame)


def work(case):
    kind = case["kind"]
    nc = case["n1"] + 27 * case["n2"]
    mlp = 2 * (32 * 64 + 64 * 64 + 64 * nc)  # operations of one decode
    shade = 2 * 28 + 2 * 27 + 40
    if kind in ("frame", "frames"):
        n = _case_cells(case).shape[0]
        rays = case["width"] * case["height"]
        count = case.get("count", 1)
        tables = 1 if case.get("one_t") else count
        rec = {"f32": 4 * nc, "bf16": 2 * nc, "f16": 2 * nc, "fp8": nc + 4, "latent": 64}[case["storage"]]
        per_leaf = 2 * nc if case["storage"] != "latent" else 2 * (32 * 64 + 64 * 64 + 64 * 28)
        seen = min(n, VISITS * rays)
        return {"bytes": tables * seen * rec + count * (12 * rays + min(4 * n, 32 * rays)),
                "flops": tables * seen * per_leaf + count * VISITS * rays * shade}
    if kind in ("rays", "finetune"):
        n = _case_cells(case).shape[0]
        hits = min(n, 14 * case["rays"])  # training rays at 800x800: more of them meet the body
        rows = 4 * nc * hits
        if kind == "rays":  # the coefficients come in and the gradients go out whole
            return {"bytes": 8 * nc * n + 52 * case["rays"], "flops": 14 * case["rays"] * (6 * nc + shade)}
        return {"bytes": 9 * rows + 52 * case["rays"], "flops": 14 * case["rays"] * (6 * nc + shade) + 12 * nc * hits}
    if kind == "dft":
        T, n = case["frames"], case["leaves"]
        return {"bytes": 4 * n * (28 * T + nc), "flops": 2 * n * T * nc}
    if kind == "latent":
        b, weights = case["batch"], 32 * 64 + 64 * 64 + 64 * nc
        return {"bytes": b * (4 * nc + 4 + 6 * 128) + 28 * weights, "flops": 3 * b * mlp + 10 * (32 * b + weights)}
    n = _case_cells(case).shape[0]
    hits = min(n, 14 * case["rays"])
    # every leaf is decoded in the general case; only the rows that rays meet are read and written
    return {"bytes": 128 * n + 12 * nc * hits + n, "flops": mlp * n + 14 * case["rays"] * (8 * nc + 2 * shade)}


def tolerance(case):
    """About four times the error against `exact` that was measured; `max` leaves room for a ray whose
    early stop, or whose grazing of a leaf's edge, is decided the other way."""
    kind = case["kind"]
    if kind in ("frame", "frames"):  # measured 3e-7 .. 9e-7 (FP32 table), 3e-6 .. 7e-6 (FP16 table)
        return {"rel": 4e-6, "max": 1e-3} if case["storage"] == "f32" else {"rel": 3e-5, "max": 5e-3}
    if kind == "rays":  # 1.3e-5 .. 2.5e-5: the colour behind a segment as a difference of FP32 sums
        return {"rel": 1e-4, "max": 0.02}
    if kind == "finetune":  # 6e-4 in m: the rows of leaves that only one of the two walks grazes
        return {"rel": 2e-3, "max": 0.15}
    if kind == "dft":  # 1.4e-7
        return {"rel": 1e-6}
    if kind == "latent":  # 5e-3 with BF16 operands; 2e-7 in FP32
        return {"rel": 2e-2, "max": 0.2} if case["tensor_cores"] else {"rel": 1e-6, "max": 1e-4}
    # 1.6e-4 with FP16 hidden activations
    return {"rel": 8e-4 if case["tensor_cores"] else 1e-4, "max": 0.05, "differ": 1e-3}


# --------------------------------------------------------------------------
# the same in FP64


def _basis(t, n):
    """Eq. 8 at times t [k]: [k, n] (cosines at even, sines at odd indices)."""
    i = torch.arange(n, device=DEV)
    f = torch.where(i % 2 == 1, i + 1, i).double()
    a = t.double()[:, None] * f[None] * (math.pi / PERIOD)
    return torch.where(i % 2 == 1, torch.sin(a), torch.cos(a))


def _sh(d):
    """Real SH of degree <= 2 at unit directions [k, 3]: [k, 9]."""
    x, y, z = d.unbind(1)
    c1, c2 = math.sqrt(3 / (4 * math.pi)), math.sqrt(15 / math.pi) / 2
    c3, c4 = math.sqrt(5 / math.pi) / 4, math.sqrt(15 / math.pi) / 4
    return torch.stack([torch.full_like(x, 0.5 / math.sqrt(math.pi)), -c1 * y, c1 * z, -c1 * x, c2 * x * y, -c2 * y * z,
                        c3 * (3 * z * z - 1), -c2 * x * z, c4 * (x * x - y * y)], 1)


def _camera_rays(cam):
    e, tg, up = (torch.tensor(v, dtype=torch.float64, device=DEV) for v in (cam.eye, cam.target, cam.up))
    f = (tg - e) / (tg - e).norm()
    r = torch.linalg.cross(f, up)
    r = r / r.norm()
    u = torch.linalg.cross(r, f)
    th = math.tan(math.radians(cam.fov_y_deg) / 2)
    py, px = torch.meshgrid(torch.arange(cam.height, device=DEV), torch.arange(cam.width, device=DEV), indexing="ij")
    sx = ((2 * (px.reshape(-1, 1).double() + 0.5) / cam.width - 1) * th) * (cam.width / cam.height)
    sy = (1 - 2 * (py.reshape(-1, 1).double() + 0.5) / cam.height) * th
    d = f + sx * r + sy * u
    return e.expand_as(d), d


def _grid(case):
    """Leaf index + 1 of every finest cell (0: empty)."""
    G = 1 << case["depth"]
    xyz = torch.as_tensor(_case_cells(case).astype(np.int64), device=DEV)
    grid = torch.zeros(G ** 3, dtype=torch.int32, device=DEV)
    grid[(xyz[:, 0] * G + xyz[:, 1]) * G + xyz[:, 2]] = torch.arange(1, xyz.shape[0] + 1, dtype=torch.int32, device=DEV)
    return grid


def _walk(grid, depth, o, d, shade, log=None):
    """Composited colour [k, 3] of the rays; shade(leaf, ray) gives (sigma_raw, colour) of a visit."""
    G = 1 << depth
    d = d.double() / d.double().norm(dim=1, keepdim=True)
    k = d.shape[0]
    C = torch.zeros((k, 3), dtype=torch.float64, device=DEV)
    T = torch.ones(k, dtype=torch.float64, device=DEV)
    go, gd = o.double() * G, d * G
    inf = torch.full_like(gd, math.inf)
    inv = torch.where(gd != 0, 1.0 / gd, inf)
    ta, tb = -go * inv, (G - go) * inv
    flat = gd == 0
    ta, tb = torch.where(flat, -inf, ta), torch.where(flat, inf, tb)
    t0 = torch.minimum(ta, tb).amax(1).clamp_min(0.0)
    t1 = torch.maximum(ta, tb).amin(1)
    ok = (t0 < t1) & ~(flat & ((go < 0) | (go > G))).any(1)
    ray = torch.nonzero(ok).flatten()
    go = (go + t0[:, None] * gd)[ray]
    gd, inv, flat = gd[ray], inv[ray], flat[ray]
    P = go.floor().long().clamp(0, G - 1)
    pos = (gd > 0).long()
    t = torch.zeros(ray.shape[0], dtype=torch.float64, device=DEV)
    alive = torch.ones_like(t, dtype=torch.bool)
    step = 0
    while ray.shape[0]:
        te = torch.where(flat, math.inf, ((P + pos).double() - go) * inv)
        tx, axis = te.min(1)
        cell = (P[:, 0] * G + P[:, 1]) * G + P[:, 2]
        hit = torch.nonzero(alive & (grid[cell] > 0) & (tx > t)).flatten()
        if hit.shape[0]:
            r, leaf, delta = ray[hit], grid[cell[hit]].long() - 1, (tx - t)[hit]
            sraw, col = shade(leaf, r)
            e = torch.exp(-sraw.clamp_min(0.0) * delta)
            Tb = T[r]
            w = Tb * (1 - e)
            C[r] += w[:, None] * col
            T[r] = Tb * e
            if log is not None:
                log.append((r, leaf, delta, sraw, col, w, Tb * e))
            alive[hit[T[r] < STOP_T]] = False
        t = torch.maximum(t, tx)
        a = axis[:, None]
        P.scatter_add_(1, a, 2 * pos.gather(1, a) - 1)
        q = P.gather(1, a).squeeze(1)
        alive &= (q >= 0) & (q < G)
        P.clamp_(0, G - 1)
        step += 1
        if step % 8 == 0:
            keep = torch.nonzero(alive).flatten()
            ray, go, gd, inv, flat, P, pos, t = (x[keep] for x in (ray, go, gd, inv, flat, P, pos, t))
            alive = alive[keep]
    return C + T[:, None] * torch.tensor(BG, dtype=torch.float64, device=DEV)


def _table(coeffs, t, n1, n2):
    """sigma_raw [n] and z [n, 27] of every leaf at time t."""
    b = _basis(torch.tensor([t], device=DEV), max(n1, n2))[0]
    sig = torch.empty(coeffs.shape[0], dtype=torch.float64, device=DEV)
    z = torch.empty((coeffs.shape[0], 27), dtype=torch.float64, device=DEV)
    for s in range(0, coeffs.shape[0], 1 << 18):
        c = coeffs[s:s + (1 << 18)].double()
        sig[s:s + (1 << 18)] = c[:, :n1] @ b[:n1]
        z[s:s + (1 << 18)] = c[:, n1:].reshape(-1, 27, n2) @ b[:n2]
    return sig, z


def _stored(c, storage):
    """The coefficients as a storage precision holds them (FP64)."""
    if storage == "bf16":
        return c.bfloat16().double()
    if storage == "f16":
        return c.half().double()
    if storage == "fp8":
        scale = c.abs().amax(1, keepdim=True) / 448.0
        return (c / scale).to(torch.float8_e4m3fn).double() * scale.double()
    return c


def _mlp(w, x):
    """Decoder outputs and hidden layers in FP64."""
    z1 = x @ w["w1"].T + w["b1"]
    h1 = z1.clamp_min(0.0)
    z2 = h1 @ w["w2"].T + w["b2"]
    h2 = z2.clamp_min(0.0)
    return h2 @ w["w3"].T + w["b3"], z1, h1, z2, h2


def _rounded(w):
    """The decoder as the tensor-core decode holds it: FP16 latents, BF16 weights."""
    return {k: (x.half() if k == "lat" else x.bfloat16() if k[0] == "w" else x).double() for k, x in w.items()}


def _exact_frames(case, seed):
    g = _gen(seed)
    n, n1, n2 = _case_cells(case).shape[0], case["n1"], case["n2"]
    cams, times = _views(case, seed)
    if case["storage"] == "latent":
        w = _rounded(_decoder(g, n, n1, n2))
        c = _mlp(w, w["lat"])[0]
    else:
        c = _stored(_coeffs(g, n, n1, n2), case["storage"])
    grid, out = _grid(case), []
    for cam, t in zip(cams, times):
        sig, z = _table(c, t, n1, n2)
        o, d = _camera_rays(cam)
        Y = _sh(d / d.norm(dim=1, keepdim=True))

        def shade(leaf, r):
            return sig[leaf], torch.sigmoid((z[leaf].reshape(-1, 3, 9) * Y[r][:, None]).sum(-1))

        out.append(_walk(grid, case["depth"], o, d, shade))
    return torch.stack(out) if case["kind"] == "frames" else out[0]


def _exact_rays(case, coeffs, o, d, t, log=None):
    n1, n2 = case["n1"], case["n2"]
    Y = _sh(d.double() / d.double().norm(dim=1, keepdim=True))
    b = _basis(t, max(n1, n2))

    def shade(leaf, r):
        c = coeffs[leaf].double()
        z = (c[:, n1:].reshape(-1, 27, n2) * b[r][:, None, :n2]).sum(-1)
        return (c[:, :n1] * b[r][:, :n1]).sum(1), torch.sigmoid((z.reshape(-1, 3, 9) * Y[r][:, None]).sum(-1))

    return _walk(_grid(case), case["depth"], o, d, shade, log)


def _exact_grad(case, rgb, dl, d, t, log, n):
    """dL/d(coefficients) [n, nc] from the logged visits, and the visited leaves."""
    n1, n2 = case["n1"], case["n2"]
    Y = _sh(d.double() / d.double().norm(dim=1, keepdim=True))
    b = _basis(t, max(n1, n2))
    grad = torch.zeros((n, n1 + 27 * n2), dtype=torch.float64, device=DEV)
    mark = torch.zeros(n, dtype=torch.uint8, device=DEV)
    P = torch.zeros_like(rgb)
    for r, leaf, delta, sraw, col, w, Tn in log:
        P[r] += w[:, None] * col
        ds = delta * (dl[r] * (Tn[:, None] * col - (rgb[r] - P[r]))).sum(1) * (sraw > 0)
        gu = dl[r] * w[:, None] * col * (1 - col)
        gz = (gu[:, :, None] * Y[r][:, None]).reshape(-1, 27, 1) * b[r][:, None, :n2]
        grad.index_add_(0, leaf, torch.cat([ds[:, None] * b[r][:, :n1], gz.reshape(-1, 27 * n2)], 1))
        mark[leaf] = 1
    return grad, mark


def _adam(p, m, v, g, lr, betas, step):
    m = betas[0] * m + (1 - betas[0]) * g
    v = betas[1] * v + (1 - betas[1]) * g * g
    return p - lr * (m / (1 - betas[0] ** step)) / ((v / (1 - betas[1] ** step)).sqrt() + EPS), m, v


def _exact_finetune(case, seed):
    c, (o, d, t, y), (m, v), _ = _fine_inputs(case, seed)
    log = []
    rgb = _exact_rays(case, c, o, d, t, log)
    diff = rgb - y.double()
    loss, dl = (diff * diff).sum(1).mean(), diff * (2.0 / case["rays"])
    if case["kind"] == "rays":
        return {"rgb": rgb, "grad": _exact_grad(case, rgb, dl, d, t, log, c.shape[0])[0]}
    grad, mark = _exact_grad(case, rgb, dl, d, t, log, c.shape[0])
    p, m, v = c.double(), m.double(), v.double()
    rows = torch.nonzero(mark).flatten()
    p[rows], m[rows], v[rows] = _adam(p[rows], m[rows], v[rows], grad[rows], LR, BETAS, FIT_STEPS + 1)
    return {"loss": loss, "param": p, "m": m, "v": v}


def _exact_dft(case, seed):
    v = _dft_values(case, seed)
    T, n, n1, n2 = case["frames"], case["leaves"], case["n1"], case["n2"]
    i = torch.arange(max(n1, n2), device=DEV)
    f = torch.where(i % 2 == 1, i + 1, i).double()
    a = torch.arange(1, T + 1, device=DEV).double()[:, None] * f[None] * (math.pi / T)
    w = torch.where(i % 2 == 1, torch.sin(a), torch.cos(a)) * torch.where(i == 0, 1.0 / T, 2.0 / T)
    out = torch.empty((n, n1 + 27 * n2), dtype=torch.float64, device=DEV)
    for s in range(0, n, 1 << 15):
        x = v[:, s:s + (1 << 15)].double()
        out[s:s + (1 << 15), :n1] = torch.einsum("tn,ti->ni", x[..., 0], w[:, :n1])
        out[s:s + (1 << 15), n1:] = torch.einsum("tnk,ti->nki", x[..., 1:], w[:, :n2]).reshape(-1, 27 * n2)
    return out


def _exact_latent(case, seed):
    w, mv, targets, rows, cw = _latent_inputs(case, seed)
    w, cw, rows = {k: x.double() for k, x in w.items()}, cw.double(), rows.long()
    x = w["lat"][rows]
    y, z1, h1, z2, h2 = _mlp(w, x)
    err = y - targets[rows].double()
    dy = 2 * cw * err
    d2 = (dy @ w["w3"]) * (z2 > 0)
    d1 = (d2 @ w["w2"]) * (z1 > 0)
    scale = 1.0 / case["batch"]
    g = {"w3": dy.T @ h2, "b3": dy.sum(0), "w2": d2.T @ h1, "b2": d2.sum(0), "w1": d1.T @ x, "b1": d1.sum(0)}
    g = {k: v * scale for k, v in g.items()}
    p, m, v = {}, {}, {}
    for k in w:
        mk, vk = mv[k][0].double(), mv[k][1].double()
        if k == "lat":
            p[k], m[k], v[k] = w[k].clone(), mk, vk
            p[k][rows], m[k][rows], v[k][rows] = _adam(x, mk[rows], vk[rows], (d1 @ w["w1"]) * scale, 1e-2, BETAS, FIT_STEPS + 1)
        else:
            p[k], m[k], v[k] = _adam(w[k], mk, vk, g[k], 1e-3, BETAS, FIT_STEPS + 1)
    return {"loss": (cw * err * err).sum().reshape(1), "p": p, "m": m, "v": v, "g": g}


def _exact_pixel(case, seed):
    g = _gen(seed)
    n, n1, n2 = _case_cells(case).shape[0], case["n1"], case["n2"]
    w = _decoder(g, n, n1, n2)
    target = _coeffs(g, n, n1, n2)
    o, d, t = camera_ray_batch(_ring(), case["rays"], _gen(seed))
    w = _rounded(w) if case["tensor_cores"] else {k: x.double() for k, x in w.items()}
    log = []
    rgb = _exact_rays(case, _mlp(w, w["lat"])[0], o, d, t, log)
    diff = rgb - _exact_rays(case, target, o, d, t)
    dy, mark = _exact_grad(case, rgb, diff * (20.0 / case["rays"]), d, t, log, n)
    return {"loss": (diff * diff).sum(1).mean(), "dy": dy, "mark": mark}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("frame", "frames"):
        return _exact_frames(case, seed)
    if kind in ("rays", "finetune"):
        return _exact_finetune(case, seed)
    if kind == "dft":
        return _exact_dft(case, seed)
    return _exact_latent(case, seed) if kind == "latent" else _exact_pixel(case, seed)
