"""What the framework is timed on: the work that its users have it do.

One training iteration of each scene type (bounded, contracted unbounded,
forward-facing), rendering without the backward, the learned proposal's
training and its render, and the single layers that a program composes
itself through the autograd functions (colour MLP, grid query, compositing
with the distortion loss).  Scenes are the synthetic ones of
paper_2206_05085_gb300.synth: blob densities, Gaussian features, seeded
cameras; the grids are drawn on the GPU here because the large ones take
seconds on the host.

Training cases use the learning rates of a late schedule (1e-4 / 1e-5), so
that the scene, and with it the number of samples in front of the halt, stays
what it is while a case is repeated, and Adam's eps = 1e-8 (torch's default),
so that a gradient at rounding level does not decide an update's sign.
"""
import dataclasses
import math

import torch

from paper_2206_05085_gb300 import _lib as L
from paper_2206_05085_gb300 import ops, synth
from paper_2206_05085_gb300.proposal import N_CAND, N_DRAW, Proposal, candidate_params
from paper_2206_05085_gb300.train import FEAT, Trainer, alpha_shift

DEV = "cuda"
T_STOP = 1e-3
ALPHA_INIT = 1e-4
GRID_LR, MLP_LR, EPS = 1e-4, 1e-5, 1e-8


def listed():
    return [
        # the smallest workload's whole iteration, eager, with the trainer's default
        # precision (colour MLP in FP32 on the CUDA cores)
        {"name": "step_small_64", "kind": "step", "scene": "bounded", "gx": 64, "gy": 64, "gz": 64, "rays": 2048,
         "precision": "f32", "graph": False, "mask_update": False, "cull": False},
        # the headline: one iteration of the 160^3 bounded scene as a replayed CUDA graph
        {"name": "step_dvgo_160", "kind": "step", "scene": "bounded", "gx": 160, "gy": 160, "gz": 160, "rays": 8192,
         "precision": "f32tc", "graph": True, "mask_update": False, "cull": False},
        # the largest: unbounded scene, 320^3 contracted grids, up to 512 samples per ray
        {"name": "step_unbounded_320", "kind": "step", "scene": "contracted", "gx": 320, "gy": 320, "gz": 320,
         "rays": 8192, "precision": "f32tc", "graph": False, "mask_update": False, "cull": False},
        # forward-facing capture: 256 depth layers of 384 x 384, one sample per layer
        {"name": "step_forward_384", "kind": "step", "scene": "forward", "gx": 384, "gy": 384, "gz": 256,
         "rays": 8192, "precision": "f32tc", "graph": False, "mask_update": False, "cull": False},
        # rendering (no backward) of 16384 rays in the BF16 form: evaluation and serving
        {"name": "render_160_bf16", "kind": "render", "scene": "bounded", "gx": 160, "gy": 160, "gz": 160,
         "rays": 16384, "precision": "bf16"},
        # colour MLP alone, forward and backward, at a training batch's live samples (odd count)
        {"name": "rgbnet_f32tc", "kind": "rgbnet", "samples": 393909, "precision": "f32tc"},
        # the same in the BF16 form at a 16384-ray batch
        {"name": "rgbnet_bf16", "kind": "rgbnet", "samples": 786433, "precision": "bf16"},
        # the smallest call: the MLP on a handful of rays, where launches and latency count
        {"name": "rgbnet_tiny", "kind": "rgbnet", "samples": 1003, "precision": "f32tc"},
        # one update of the learned proposal: 16384 rays, up to 512 candidates each
        {"name": "proposal_train", "kind": "proposal_train", "gx": 160, "gy": 160, "gz": 160, "rays": 16384},
        # a render through the proposal: candidates, picks, at most 64 samples per ray
        {"name": "proposal_render", "kind": "proposal_render", "gx": 160, "gy": 160, "gz": 160, "rays": 4099,
         "precision": "f32tc"},
        # trilinear queries of both grids and their adjoints through autograd
        {"name": "query_160", "kind": "query", "gx": 160, "gy": 160, "gz": 160, "samples": 762026},
        # compositing and distortion loss over ragged rays, forward and backward, through autograd
        {"name": "composite_8192", "kind": "composite", "rays": 8192, "mean": 93},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "render", "rgbnet", "rgbnet", "proposal_train", "proposal_render",
                       "query", "composite"])
    prec = rng.choice(["f32tc", "f32tc", "bf16", "f32"])
    dims = [rng.randint(48, 200) for _ in range(3)]
    box = dict(zip(("gx", "gy", "gz"), dims))
    if kind == "step":
        scene = rng.choice(["bounded", "bounded", "contracted", "forward"])
        if scene == "contracted":
            g = rng.randint(96, 300)
            box = {"gx": g, "gy": g, "gz": g}
        elif scene == "forward":
            box = {"gx": rng.randint(96, 340), "gy": rng.randint(96, 340), "gz": rng.randint(48, 200)}
        rays = _log(rng, 256, 8192 if scene == "contracted" else 16384)
        return {"kind": kind, "scene": scene, **box, "rays": rays, "precision": prec,
                "graph": rng.random() < 0.5, "mask_update": scene != "contracted" and rng.random() < 0.3,
                "cull": rng.random() < 0.2}
    if kind == "render":
        return {"kind": kind, "scene": "bounded", **box, "rays": _log(rng, 1024, 40000), "precision": prec}
    if kind == "rgbnet":
        return {"kind": kind, "samples": _log(rng, 200, 900000), "precision": prec}
    if kind == "proposal_train":
        return {"kind": kind, **box, "rays": _log(rng, 512, 16384)}
    if kind == "proposal_render":
        return {"kind": kind, **box, "rays": _log(rng, 512, 16384), "precision": rng.choice(["f32tc", "bf16"])}
    if kind == "query":
        return {"kind": kind, **box, "samples": _log(rng, 2000, 1500000)}
    return {"kind": kind, "rays": _log(rng, 256, 20000), "mean": rng.randint(3, 300)}


# ------------------------------------------------------------------ scenes
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _config(case):
    scene, dims = case.get("scene", "bounded"), (case["gx"], case["gy"], case["gz"])
    base = {"bounded": synth.CFG2, "contracted": synth.CFG3, "forward": synth.CFG6}[scene]
    if scene == "bounded" and dims == (64, 64, 64):
        base = synth.CFG1
    cfg = dataclasses.replace(base, grid=dims[0], dims=dims, n_rays=case["rays"])
    # the mean voxel size sets the sampling step of a non-cubic box
    mean = int(round(sum(dims) / 3))
    rp = synth.render_params(dataclasses.replace(cfg, grid=mean) if scene != "forward" else cfg)
    return cfg, dataclasses.replace(rp, lr_grid=GRID_LR, lr_mlp=MLP_LR, eps=EPS)


def _grids(cfg, seed):
    """Density [Z, Y, X] and features [Z, Y, X, C] of the config's recipe, on the GPU."""
    g = _gen(seed)
    gx, gy, gz = cfg.dims
    ax = [torch.linspace(cfg.bbox_min, cfg.bbox_max, n, device=DEV) for n in (gz, gy, gx)]
    Z, Y, X = ax[0].view(-1, 1, 1), ax[1].view(1, -1, 1), ax[2].view(1, 1, -1)
    c = (torch.rand(cfg.n_blobs, 3, generator=g, device=DEV) * 2 - 1) * cfg.blob_center_range
    s = cfg.sigma_lo + (cfg.sigma_hi - cfg.sigma_lo) * torch.rand(cfg.n_blobs, generator=g, device=DEV)
    c, s = c.tolist(), s.tolist()
    D = torch.randn(gz, gy, gx, generator=g, device=DEV) * cfg.noise_std + cfg.blob_bias
    for (bx, by, bz), sb in zip(c, s):
        k = -0.5 / (sb * sb)
        D += (cfg.blob_peak - cfg.blob_bias) * (torch.exp(k * (X - bx) ** 2) * torch.exp(k * (Y - by) ** 2)
                                                * torch.exp(k * (Z - bz) ** 2))
    if cfg.shell is not None:
        lo, hi, raw = cfg.shell
        r = torch.maximum(torch.maximum(X.abs(), Y.abs()), Z.abs())
        D = torch.where((r >= lo) & (r <= hi), D.clamp(min=raw), D)
    F = torch.randn(gz, gy, gx, FEAT, generator=g, device=DEV) * cfg.feat_std
    return D, F


def _rays(cfg, seed):
    o, d = synth.rays(cfg, seed=seed)
    t = synth.target_rgb(cfg, seed=seed)
    return tuple(torch.from_numpy(a).to(DEV) for a in (o, d, t))


def _trainer(case, cfg, rp, seed, **kw):
    D, F = _grids(cfg, seed)
    return Trainer(cfg, rp, D.cpu().numpy(), F.cpu().numpy(), synth.mlp_params(seed=seed), cfg.n_rays,
                   precision=case.get("precision", "f32tc"), device=DEV, **kw)


def _ragged(rays, mean, g):
    """ray_off of a ragged batch: a fifth of the rays empty, the rest spread around their mean
    (the same lengths for every seed, in another order)."""
    n = ((torch.arange(rays, device=DEV) * 0.618034) % 1.0 * 2 * mean * 1.25).long()
    n[4::5] = 0
    n[0] = max(1, mean)
    n = n[torch.randperm(rays, generator=g, device=DEV)]
    return torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), n.cumsum(0)])


# ----------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "render"):
        cfg, rp = _config(case)
        kw = {}
        if kind == "step":
            kw = {"mask_update": case["mask_update"], "w_min": 1e-4 if case["cull"] else None}
        tr = _trainer(case, cfg, rp, seed, **kw)
        st = {"kind": kind, "tr": tr, "rays": _rays(cfg, seed)}
        if kind == "step" and case["graph"]:
            st["graph"], st["inputs"] = tr.capture(*st["rays"])
        return st
    if kind in ("proposal_train", "proposal_render"):
        cfg, rp = _config(case)
        rp_c = candidate_params(cfg, rp)
        tr = _trainer(case, cfg, dataclasses.replace(rp_c, max_steps=N_DRAW), seed)
        grid, dt = tr.density.render_view
        prop = Proposal(cfg, rp, grid, dt, synth.proposal_params(seed), cfg.n_rays, lr=1e-3)
        return {"kind": kind, "tr": tr, "prop": prop, "rays": _rays(cfg, seed)}
    if kind == "rgbnet":
        return {"kind": kind, "precision": case["precision"], **_mlp_inputs(case, seed)}
    if kind == "query":
        q = _query_inputs(case, seed)
        G = (case["gx"], case["gy"], case["gz"])
        gd = L.GridDesc.make(-1.0, 1.0, G)
        packed = []
        for dense, C in ((q["D"], 1), (q["F"], FEAT)):
            p = torch.empty(L.grid_bricked_elems(G, C), device=DEV)
            L.grid_pack(dense, p, G, C, L.F32)
            packed.append(p.requires_grad_())
        return {"kind": kind, "gd": gd, "density": packed[0], "feature": packed[1],
                **{k: q[k] for k in ("xyz", "g_raw", "g_k0")}}
    return {"kind": kind, **_composite_inputs(case, seed)}


def _mlp_inputs(case, seed):
    """Features, directions and upstream gradients of a live-sample list: ~50
    consecutive samples per ray, gradients w * g_color with w from 1e-5 to 1."""
    g, n = _gen(seed), case["samples"]
    rays = n // 50 + 1
    d = torch.randn(rays, 3, generator=g, device=DEV)
    d = d / d.norm(dim=1, keepdim=True)
    ray_id = torch.sort(torch.randint(rays, (n,), generator=g, device=DEV, dtype=torch.int32))[0]
    k0 = torch.randn(n, FEAT, generator=g, device=DEV) * 0.3
    w = torch.exp(torch.rand(n, 1, generator=g, device=DEV) * math.log(1e-5))
    g_rgb = w * torch.randn(n, 3, generator=g, device=DEV) / rays
    params = torch.from_numpy(synth.mlp_params(seed=seed)).to(DEV)
    return {"k0": k0.requires_grad_(), "params": params.requires_grad_(), "d": d, "ray_id": ray_id, "g_rgb": g_rgb}


def _query_inputs(case, seed):
    """Points along rays through the box (half-voxel steps, as the samplers
    make them), the grids and upstream gradients."""
    cfg = dataclasses.replace(synth.CFG2, grid=case["gx"], dims=(case["gx"], case["gy"], case["gz"]))
    D, F = _grids(cfg, seed)
    g, n = _gen(seed + 1), case["samples"]
    per, step = 93, 1.0 / max(cfg.dims)
    rays = (n + per - 1) // per
    mid = (torch.rand(rays, 1, 3, generator=g, device=DEV) * 2 - 1) * 0.6
    d = torch.randn(rays, 1, 3, generator=g, device=DEV)
    d = d / d.norm(dim=2, keepdim=True)
    t = (torch.arange(per, device=DEV) - per / 2).view(1, per, 1) * step
    xyz = (mid + t * d).reshape(-1, 3)[:n].contiguous()
    return {"D": D, "F": F, "xyz": xyz, "g_raw": torch.randn(n, 1, generator=g, device=DEV) * 1e-4,
            "g_k0": torch.randn(n, FEAT, generator=g, device=DEV) * 1e-5}


def _composite_inputs(case, seed):
    """Raw densities of rays that pass through empty space into a blob, colours,
    midpoints and lengths of the samples, upstream gradients."""
    g, R = _gen(seed), case["rays"]
    off = _ragged(R, case["mean"], g)
    S = int(off[-1])
    ray = torch.repeat_interleave(torch.arange(R, device=DEV), off[1:] - off[:-1])
    n = (off[1:] - off[:-1])[ray].float()
    m = (torch.arange(S, device=DEV) - off[ray] + 0.5) / n
    centre = 0.2 + 0.6 * torch.rand(R, generator=g, device=DEV)[ray]
    width = 0.05 + 0.15 * torch.rand(R, generator=g, device=DEV)[ray]
    peak = 14 * torch.rand(R, generator=g, device=DEV)[ray]
    raw = -4 + peak * torch.exp(-0.5 * ((m - centre) / width) ** 2)
    raw = raw + 0.1 * torch.randn(S, generator=g, device=DEV)
    return {"raw": raw.requires_grad_(), "rgb": torch.rand(S, 3, generator=g, device=DEV).requires_grad_(),
            "off": off, "m": m, "ds": 1.0 / n, "g_color": torch.randn(R, 3, generator=g, device=DEV) / R,
            "g_L": torch.full((R,), 0.01 / R, device=DEV)}


# --------------------------------------------------------------------- run
def run(st):
    kind = st["kind"]
    if kind == "step":
        tr = st["tr"]
        if "graph" in st:
            for dst, src in zip(st["inputs"], st["rays"]):   # the batch enters the graph's buffers
                dst.copy_(src)
            st["graph"].replay()
        else:
            tr.step(*st["rays"])
        return {"loss": tr.loss, "color": tr.color, "mlp": tr.mlp, "mlp_m": tr.mlp_m,
                "density": tr.density.p, "density_m": tr.density.m, "feature": tr.feature.p, "feature_m": tr.feature.m}
    if kind == "render":
        tr = st["tr"]
        tr.forward(*st["rays"])
        return {"color": tr.color, "loss": tr.loss, "T_end": tr.T_end, "n_live": tr.n_live, "ray_off": tr.ray_off}
    if kind == "proposal_train":
        p = st["prop"]
        loss = p.train_step(*st["rays"][:2])
        return {"loss": loss, "params": p.params, "m": p.m}
    if kind == "proposal_render":
        p, tr = st["prop"], st["tr"]
        o, d, t = st["rays"]
        p.select_into(tr, o, d)
        tr.forward(o, d, t, sample=False)
        return {"color": tr.color, "loss": tr.loss, "ray_off": tr.ray_off, "n_sel": p.n_sel, "sel": p.sel}
    if kind == "rgbnet":
        rgb = ops.rgbnet(st["k0"], st["params"], st["d"], st["ray_id"], st["precision"])
        g_k0, g_params = torch.autograd.grad(rgb, (st["k0"], st["params"]), st["g_rgb"])
        return {"rgb": rgb.detach(), "g_k0": g_k0, "g_params": g_params}
    if kind == "query":
        raw = ops.sample_grid(st["density"], st["xyz"], st["gd"], 1)
        k0 = ops.sample_grid(st["feature"], st["xyz"], st["gd"], FEAT)
        g = torch.autograd.grad((raw, k0), (st["density"], st["feature"]), (st["g_raw"], st["g_k0"]))
        return {"raw": raw.detach(), "k0": k0.detach(), "g_density": g[0], "g_feature": g[1]}
    color, w, n_live = ops.composite(st["raw"], st["rgb"], st["off"], alpha_shift(ALPHA_INIT), 0.5, T_STOP,
                                     (1.0, 1.0, 1.0))
    L_r = ops.distortion(w, st["m"], st["ds"], st["off"], n_live)
    g_raw, g_rgb = torch.autograd.grad((color, L_r), (st["raw"], st["rgb"]), (st["g_color"], st["g_L"]))
    return {"color": color.detach(), "w": w.detach(), "n_live": n_live, "L_r": L_r.detach(), "g_raw": g_raw,
            "g_rgb": g_rgb}


# -------------------------------------------------------------------- work
MLP_FLOP = 2 * (39 * 128 + 128 * 128 + 128 * 3)
PROP_FLOP = 2 * (39 * 64 + 64 * 64 + 64)


def _live(case):
    """Samples in front of the halt per batch, as counted on the listed scenes
    (8192 rays: 160^3 4.3e5, contracted 320^3 1.9e6, 256 layers 3.6e5)."""
    mean = (case["gx"] + case["gy"] + case["gz"]) / 3
    per = {"bounded": 0.33 * mean, "contracted": 0.72 * mean, "forward": 0.17 * case["gz"]}[case.get("scene", "bounded")]
    return case["rays"] * per


def work(case):
    """Inputs read once, outputs written once: rays, the grid voxels a batch
    reaches (about two distinct ones per live sample, both grids), weights."""
    kind = case["kind"]
    if kind in ("step", "render"):
        live = _live(case)
        vox = min(2 * live, 0.25 * case["gx"] * case["gy"] * case["gz"])
        value = 26 if case["precision"] == "bf16" else 52
        if kind == "render":
            return {"bytes": 48 * case["rays"] + value * vox, "flops": live * MLP_FLOP}
        # p, m and v of both grids in and out once per reached voxel
        return {"bytes": 48 * case["rays"] + 6 * 52 * vox, "flops": 3 * live * MLP_FLOP}
    if kind == "proposal_train":
        cand = 0.65 * N_CAND * case["rays"]
        return {"bytes": 28 * case["rays"] + 4 * case["gx"] * case["gy"] * case["gz"], "flops": 3 * cand * PROP_FLOP}
    if kind == "proposal_render":
        cand = 0.65 * N_CAND * case["rays"]
        picks = 0.8 * N_DRAW * case["rays"]
        return {"bytes": 48 * case["rays"] + 52 * min(8 * picks, case["gx"] * case["gy"] * case["gz"]),
                "flops": cand * PROP_FLOP + picks * MLP_FLOP}
    if kind == "rgbnet":
        n = case["samples"]
        return {"bytes": n * (2 * 4 * FEAT + 4 + 2 * 12) + 12 * (n // 50), "flops": 3 * n * MLP_FLOP}
    if kind == "query":
        n, vox = case["samples"], case["gx"] * case["gy"] * case["gz"]
        # positions, outputs and upstream rows; each reached voxel read; both gradients written whole
        return {"bytes": n * (12 + 2 * 52) + 52 * min(2 * n, vox) + 52 * vox, "flops": 2 * 2 * 8 * 13 * n}
    S = case["rays"] * case["mean"]
    return {"bytes": S * (4 + 12 + 4 + 4 + 4 + 4 + 12) + 48 * case["rays"], "flops": 60 * S}


# ------------------------------------------------------------------- exact
def exact(case, seed):
    """The layers in 64-bit torch.  The whole calls have no such value here:
    which samples exist is decided by 32-bit comparisons of the samplers, and a
    trained state follows from them."""
    kind = case["kind"]
    if kind == "rgbnet":
        return _exact_mlp(case, seed)
    if kind == "query":
        return _exact_query(case, seed)
    if kind == "composite":
        return _exact_composite(case, seed)
    return None


def _exact_mlp(case, seed):
    a = _mlp_inputs(case, seed)
    p = a["params"].detach()
    if case["precision"] == "bf16":   # this form's stored values
        p = p.to(torch.bfloat16)
    p = p.double().requires_grad_()
    sizes = [(128, 39), (128,), (128, 128), (128,), (3, 128), (3,)]
    W, at = [], 0
    for s in sizes:
        W.append(p[at:at + math.prod(s)].view(s))
        at += math.prod(s)
    g_p, rgb, g_k0 = torch.zeros_like(p), [], []
    for b in range(0, case["samples"], 1 << 17):
        e = slice(b, b + (1 << 17))
        k0 = a["k0"].detach()[e].double().requires_grad_()
        d = a["d"].double()[a["ray_id"][e].long()]
        arg = (d[:, :, None] * (2.0 ** torch.arange(4, device=DEV, dtype=torch.float64))).flatten(1)
        x = torch.cat([k0, d, arg.sin(), arg.cos()], 1)
        h = torch.relu(torch.relu(x @ W[0].T + W[1]) @ W[2].T + W[3])
        y = torch.sigmoid(h @ W[4].T + W[5])
        gk, gp = torch.autograd.grad(y, (k0, p), a["g_rgb"][e].double(), retain_graph=True)
        rgb.append(y.detach())
        g_k0.append(gk)
        g_p += gp
    return {"rgb": torch.cat(rgb), "g_k0": torch.cat(g_k0), "g_params": g_p}


def _bricked(dense, G):
    """[Z, Y, X, C] to 8^3 bricks in raster order, Morton order inside, channels innermost."""
    gx, gy, gz = G
    nb = [(n + 7) // 8 for n in G]
    C = dense.shape[-1]
    full = torch.zeros(8 * nb[2], 8 * nb[1], 8 * nb[0], C, dtype=dense.dtype, device=dense.device)
    full[:gz, :gy, :gx] = dense
    bits = full.view(nb[2], 2, 2, 2, nb[1], 2, 2, 2, nb[0], 2, 2, 2, C)
    # axes: z 0 (1 2 3), y 4 (5 6 7), x 8 (9 10 11); each axis' bits from high to low
    return bits.permute(0, 4, 8, 1, 5, 9, 2, 6, 10, 3, 7, 11, 12).reshape(-1)


def _exact_query(case, seed):
    q = _query_inputs(case, seed)
    G = (case["gx"], case["gy"], case["gz"])
    dim = torch.tensor(G, device=DEV)
    u = ((q["xyz"].double() + 1.0) * 0.5 * (dim - 1)).clamp(min=0)
    u = torch.minimum(u, (dim - 1).double())
    i = torch.minimum(u.floor().long(), dim - 2)
    f = u - i
    out = {}
    for name, dense, up, C in (("raw", q["D"][..., None], q["g_raw"], 1), ("k0", q["F"], q["g_k0"], FEAT)):
        flat, val = dense.reshape(-1, C), 0.0
        grad = torch.zeros(flat.shape, dtype=torch.float64, device=DEV)
        for k in range(8):
            o = torch.tensor([k & 1, (k >> 1) & 1, k >> 2], device=DEV)
            w = torch.where(o.bool(), f, 1 - f).prod(1, keepdim=True)
            c = i + o
            at = (c[:, 2] * G[1] + c[:, 1]) * G[0] + c[:, 0]
            val = val + w * flat[at].double()
            grad.index_add_(0, at, w * up.double())
        out[name] = val
        out["g_density" if C == 1 else "g_feature"] = _bricked(grad.view(*dense.shape[:3], C), G)
    return out


def _exact_composite(case, seed):
    a = _composite_inputs(case, seed)
    off = a["off"]
    R, n = case["rays"], off[1:] - off[:-1]
    N, S = int(n.max()), int(off[-1])
    ray = torch.repeat_interleave(torch.arange(R, device=DEV), n)
    at = torch.arange(S, device=DEV) - off[ray]

    def pad(v, fill=0.0):
        full = torch.full((R, N) + tuple(v.shape[1:]), fill, dtype=torch.float64, device=DEV)
        full[ray, at] = v.detach().double()
        return full

    raw, rgb = pad(a["raw"]).requires_grad_(), pad(a["rgb"]).requires_grad_()
    m, ds = pad(a["m"]), pad(a["ds"])
    there = pad(torch.ones(S, device=DEV)) > 0
    la = torch.where(there, -0.5 * torch.nn.functional.softplus(raw + alpha_shift(ALPHA_INIT)), 0.0)
    incl = la.cumsum(1)
    logT = torch.cat([torch.zeros(R, 1, dtype=torch.float64, device=DEV), incl[:, :-1]], 1)
    live = there & (logT.detach() >= math.log(T_STOP))
    w = torch.where(live, logT.exp() * -torch.expm1(la), 0.0)
    T_end = torch.where(live, la, 0.0).sum(1, keepdim=True).exp()
    color = (w[..., None] * rgb).sum(1) + T_end
    W, WM = w.cumsum(1) - w, (w * m).cumsum(1) - w * m
    L_r = (2 * w * (m * W - WM) + w * w * ds / 3).sum(1)
    g = torch.autograd.grad((color, L_r), (raw, rgb), (a["g_color"].double(), a["g_L"].double()))
    return {"color": color.detach(), "w": w.detach()[ray, at], "n_live": None, "L_r": L_r.detach(),
            "g_raw": g[0][ray, at], "g_rgb": g[1][ray, at]}
