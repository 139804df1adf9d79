"""The work this library is timed on: one case per call (or short chain of calls) a user's program makes.

A case is a dict: `op` names the call, the rest are its sizes and options.

  raster         autograd rendering, forward and backward (binding.rasterize)
  train          one training step (training.TrainState.step)
  query          one open-vocabulary query render: project, bin, composite, relevancy
  decode         decoder inference of a rendered view (class map and probabilities)
  decode_train   decoder training call: loss, input gradients, weight gradients
  export         language feature map of a view
  quantize       quantisation of language features against a codebook
  quantize_grad  the codebook's gradient
  smooth         adaptive spatial smoothing, loss and gradients
  densify        clone / split / prune of the Gaussians and their Adam moments

Scenes, decoders and features follow paper_2311_18482_gb300/synth.py's distributions, drawn on the GPU.
"""
import math

import numpy as np
import torch

import paper_2311_18482_gb300 as leg
from paper_2311_18482_gb300 import synth
from paper_2311_18482_gb300.training import TrainState

DEV = "cuda"
D, D_CLIP = 896, 512                       # hybrid language feature: 512 CLIP + 384 DINO dims
FIELDS = ("means", "log_scales", "quats", "opacity_raw", "sh", "feat", "unc")
DEC = ("W1", "b1", "W2", "b2", "W3", "b3")
SMO = ("W1", "b1", "W2", "b2", "W3", "b3", "W4", "b4")


def listed():
    return [
        # a toy scene or a unit test of a user's own: every launch and every host microsecond counts
        dict(name="raster_2k", op="raster", n=2000, w=128, h=128, degree=0),
        # a user's own training loop around the autograd entry, at a full capture's size
        dict(name="raster_1m", op="raster", n=1_000_000, w=1296, h=840, degree=3),
        # early training (few Gaussians, a downscaled view) with the full RGB loss
        dict(name="train_100k_dssim", op="train", n=100_000, w=640, h=480, codes=128, rgb_loss="l1_dssim"),
        # the steady state of training a full capture
        dict(name="train_1m", op="train", n=1_000_000, w=1296, h=840, codes=128, rgb_loss="l1"),
        # an interactive text query on a large scene in Full HD
        dict(name="query_3m", op="query", n=3_000_000, w=1920, h=1080, codes=256, prompts=4),
        # the class map of a small, ragged preview
        dict(name="decode_333x217", op="decode", pixels=333 * 217, hidden=64, codes=64),
        # training the published decoder widths (8-128-256-N) on a full view
        dict(name="decode_train_wide", op="decode_train", pixels=1296 * 840, hidden=128, codes=128),
        # writing a view's language features out for another program
        dict(name="export_view", op="export", pixels=1296 * 840, codes=256),
        # the index map of a full view's features: the preprocessing pass over a capture
        dict(name="quantize_view", op="quantize", features=1296 * 840, codes=128),
        # a codebook update on a smaller view whose masked pixels are left out
        dict(name="quantize_grad_300k", op="quantize_grad", features=300_007, codes=128),
        # the smoothing term of a training step at full size
        dict(name="smooth_1m", op="smooth", n=1_000_000),
        # density control of a scene that still grows
        dict(name="densify_1m", op="densify", n=1_000_000, degree=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("raster", "train", "query", "decode", "decode_train", "export", "quantize", "quantize_grad",
                     "smooth", "densify"))
    c = dict(op=op)
    if op in ("raster", "train", "query"):
        c["n"] = _log(rng, 1000, 3_000_000 if op == "query" else 1_000_000)
        c["w"] = _log(rng, 100, 1920 if op == "query" else 1296)
        c["h"] = max(64, min(1080 if op == "query" else 840, int(c["w"] * rng.uniform(0.5, 0.8))))
    if op == "raster":
        c["degree"] = rng.randint(0, 3)
    if op == "train":
        c["rgb_loss"] = rng.choice(("l1", "l1_dssim"))
    if op in ("train", "decode_train", "quantize", "quantize_grad"):
        c["codes"] = rng.choice((32, 64, 128))
    if op in ("decode", "export"):
        c["codes"] = rng.choice((32, 64, 128, 256))
    if op == "query":
        c["codes"] = rng.choice((64, 128, 192, 256))
        c["prompts"] = rng.randint(1, 8)
    if op in ("decode", "decode_train", "export"):
        c["pixels"] = _log(rng, 10_000, 1296 * 840)
    if op in ("decode", "decode_train"):
        c["hidden"] = rng.choice((64, 128))
    if op in ("quantize", "quantize_grad"):
        c["features"] = _log(rng, 10_000, 1296 * 840)
    if op in ("smooth", "densify"):
        c["n"] = _log(rng, 1000, 1_000_000)
    if op == "densify":
        c["degree"] = rng.randint(0, 3)
    return c


# ------------------------------------------------------------------------------------------------ inputs
class _Draw:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEV)

    def uniform(self, lo, hi, *shape):
        return torch.rand(shape, generator=self.g, device=DEV) * (hi - lo) + lo

    def integers(self, hi, *shape):
        return torch.randint(0, hi, shape, generator=self.g, device=DEV)


def _scene(r, n, degree):
    """Gaussians: a uniform cube up to 5,000, clusters above."""
    if n <= 5000:
        means = r.uniform(-1, 1, n, 3)
    else:
        k = 20 if n <= 200_000 else 50
        centres = r.uniform(-2, 2, k, 3)
        means = (centres[r.integers(k, n)] + 0.25 * r.normal(n, 3)).clamp(-2, 2)
    sh = 0.1 * r.normal(n, (degree + 1) ** 2, 3)
    if degree == 0:
        sh = r.uniform(-math.sqrt(math.pi), math.sqrt(math.pi), n, 1, 3)
    q = r.normal(n, 4)
    return dict(means=means, log_scales=0.5 * r.normal(n, 3) - 3, quats=q / q.norm(dim=1, keepdim=True),
                opacity_raw=r.normal(n), sh=sh, feat=r.normal(n, 8), unc=r.uniform(0, 1, n))


def _camera(case, seed):
    return synth.circle_pose(seed % 16, 16, case["w"], case["h"])


def _linear(r, *widths):
    """Weights and biases of a chain of linear layers, U(-1/sqrt(in), 1/sqrt(in))."""
    out = []
    for i, o in zip(widths, widths[1:]):
        out += [r.uniform(-1, 1, o, i) / math.sqrt(i), r.uniform(-1, 1, o) / math.sqrt(i)]
    return out


def _decoder(r, hidden, codes, sharp=1.0):
    """sharp > 1: a trained decoder's peaked class distribution."""
    w = _linear(r, 8, hidden, 2 * hidden, codes)
    w[4] *= sharp
    return w


def _voronoi(r, w, h, codes, regions=30):
    """Class map: every pixel takes the code of its nearest of a few random points."""
    sx, sy, code = r.uniform(0, w, regions), r.uniform(0, h, regions), r.integers(codes, regions)
    x, y = torch.arange(w, device=DEV), torch.arange(h, device=DEV)
    best, arg = torch.full((h, w), math.inf, device=DEV), torch.zeros((h, w), dtype=torch.int64, device=DEV)
    for k in range(regions):
        d = (x[None] - sx[k]) ** 2 + (y[:, None] - sy[k]) ** 2
        arg[d < best] = k
        best = torch.minimum(best, d)
    return code[arg].to(torch.int32), arg


def _pixels(r, n, codes):
    """Rendered compact features, uncertainties and class targets of n pixels in regions."""
    w = max(1, int(math.sqrt(1.5 * n)))
    target, region = _voronoi(r, w, -(-n // w), codes)
    region = region.reshape(-1)[:n]
    feat = (r.normal(30, 8)[region] + 0.2 * r.normal(n, 8)).t().contiguous()
    return feat, r.uniform(0, 0.5, n), target.reshape(-1)[:n].contiguous()


def _unit(x):
    return x / x.norm(dim=-1, keepdim=True)


def _features(r, k, codes):
    """Language features of a view in BF16, around one hidden code per region; a codebook of some of them."""
    w = max(1, int(math.sqrt(1.5 * k)))
    centres = torch.cat([_unit(r.normal(128, D_CLIP)), _unit(r.normal(128, D - D_CLIP))], 1)
    lab = _voronoi(r, w, -(-k // w), 128, 60)[0].reshape(-1)[:k].long()
    f = torch.empty((k, D), dtype=torch.bfloat16, device=DEV)
    for i in range(0, k, 1 << 18):
        part = lab[i:i + (1 << 18)]
        f[i:i + (1 << 18)] = centres[part] + 0.6 / math.sqrt(D) * r.normal(len(part), D)
    book = f[r.integers(k, codes)].float() + 0.1 / math.sqrt(D) * r.normal(codes, D)
    return f, book


def _numpy_scene(s, degree):
    return synth.Scene(*(s[f].cpu().numpy() for f in FIELDS), degree)


def _upstream(r, h, w):
    return [r.normal(3, h, w) / (3 * h * w), r.normal(8, h, w) / (h * w), r.normal(h, w) / (h * w)]


def _inputs(case, seed):
    """What the case's call is given: the same tensors for the library and for exact()."""
    r, op, x = _Draw(seed), case["op"], {}
    if op in ("raster", "train", "query"):
        x["cam"] = _camera(case, seed)
        x["scene"] = _scene(r, case["n"], case.get("degree", 3))
        h, w = case["h"], case["w"]
    if op == "raster":
        x["up"] = _upstream(r, h, w)
    elif op == "train":
        x["dec"] = _decoder(r, 64, case["codes"])
        x["target"] = _voronoi(r, w, h, case["codes"])[0]
        yy, xx = torch.arange(h, device=DEV)[:, None] / h, torch.arange(w, device=DEV)[None] / w
        k = r.uniform(-6, 6, 3, 4, 2) * 2 * math.pi
        ph = r.uniform(0, 2 * math.pi, 3, 4)
        x["rgb"] = (0.5 + 0.125 * torch.stack([sum(torch.sin(k[c, j, 0] * xx + k[c, j, 1] * yy + ph[c, j])
                                                   for j in range(4)) for c in range(3)])).clamp(0, 1).contiguous()
    elif op == "query":
        x["dec"] = _decoder(r, 64, case["codes"], 4.0)
        x["book"] = _unit(r.normal(case["codes"], D))
        x["text"], x["negs"] = _unit(r.normal(case["prompts"], D_CLIP)), _unit(r.normal(4, D_CLIP))
    elif op in ("decode", "decode_train", "export"):
        x["feat"], x["unc"], x["target"] = _pixels(r, case["pixels"], case["codes"])
        x["dec"] = _decoder(r, case.get("hidden", 64), case["codes"], 1.0 if op == "decode_train" else 4.0)
        if op == "export":
            x["book"] = _unit(r.normal(case["codes"], D))
    elif op in ("quantize", "quantize_grad"):
        x["f"], x["book"] = _features(r, case["features"], case["codes"])
        if op == "quantize_grad":
            b = x["book"].bfloat16()
            bc, bd = _unit(b[:, :D_CLIP].float()).bfloat16(), _unit(b[:, D_CLIP:].float()).bfloat16()
            count = torch.zeros(case["codes"], device=DEV)
            for part in x["f"].split(1 << 18):
                a, c = part[:, :D_CLIP], part[:, D_CLIP:]
                m = (_unit(a.float()).bfloat16() @ bc.t() + 0.5 * (_unit(c.float()).bfloat16() @ bd.t())).argmax(1)
                count += torch.bincount(m, minlength=case["codes"])
            x["r"] = count / case["features"]
    elif op == "smooth":
        x["scene"] = _scene(r, case["n"], 0)
        x["mlp"] = _linear(r, 3, 128, 128, 128, 8)
    elif op == "densify":
        n = case["n"]
        x["scene"] = _scene(r, n, case["degree"])
        x["m"] = {f: 1e-6 * r.normal(*t.shape) for f, t in x["scene"].items()}
        x["v"] = {f: 1e-12 * r.uniform(0, 1, *t.shape) for f, t in x["scene"].items()}
        # 10 % pruned (too large on screen, or transparent), 24 % grow, the rest stays: fixed counts, random places
        rank = torch.randperm(n, generator=r.g, device=DEV)
        prune, grow = rank < n // 10, (rank >= n // 10) & (rank < n // 3)
        big = prune & (rank % 2 == 0)
        x["scene"]["opacity_raw"] = torch.where(prune & ~big, -6.0, x["scene"]["opacity_raw"].clamp_min(-5))
        x["scene"]["log_scales"].clamp_(max=-1)
        x["radius"] = torch.where(big, r.uniform(21, 60, n), r.uniform(0, 20, n)).to(torch.int32)
        x["cnt"] = (1 + r.integers(10, n)).to(torch.int32)        # steps each Gaussian was seen on
        x["acc"] = x["cnt"] * 0.0002 * torch.where(grow, r.uniform(1.1, 4, n), r.uniform(0, 0.9, n))
        x["noise"] = r.normal(n, 2, 3)
    return x


DENSIFY = dict(grad_thresh=0.0002, percent_dense=0.01, scene_extent=4.0, min_opacity=0.005, max_screen_size=20.0,
               world_frac=0.1)


def _gaussians(s, degree):
    return leg.Gaussians(*(s[f] for f in FIELDS), degree)


def _bytes(n):
    return torch.empty(max(n, 1), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    x, op = _inputs(case, seed), case["op"]
    x["op"] = op
    if op == "raster":
        x["degree"] = case["degree"]
        x["leaves"] = [x["scene"][f].requires_grad_() for f in FIELDS]
    elif op == "train":
        st = TrainState(_numpy_scene(x.pop("scene"), 3), synth.Decoder(*(t.cpu().numpy() for t in x.pop("dec"))),
                        case["w"], case["h"], DEV, rgb_loss=case["rgb_loss"])
        st.load_state_dict(_moments(st.params, seed))
        x["st"] = st
    elif op == "query":
        n, p = case["n"], case["w"] * case["h"]
        x["g"] = _gaussians(x.pop("scene"), 3)
        x["proj"], x["bins"] = leg.Projected.empty(n), leg.BinSortBuffers()
        x["img"] = leg.Image.empty(case["h"], case["w"])
        x["ws"] = _bytes(leg.le_query_workspace(leg.FUSED_BF16, p, case["codes"], D_CLIP))
        x["out"] = torch.empty((case["prompts"], p), device=DEV)
    elif op in ("decode", "decode_train"):
        mode = leg.FUSED_BF16 | (leg.DECODE_TRAIN if op == "decode_train" else 0)
        x["ws"] = _bytes(leg.le_decode_workspace(mode, case["pixels"], leg.decoder_struct(*x["dec"])))
    elif op == "export":
        x["out"] = torch.empty((case["pixels"], D), dtype=torch.bfloat16, device=DEV)
    elif op == "quantize":
        x["ws"] = _bytes(leg.le_quantize_workspace(case["codes"], D))
    elif op == "quantize_grad":
        x["ws"] = _bytes(leg.le_quantize_grad_workspace(case["features"], case["codes"], D))
    elif op == "densify":
        x["g"], x["gm"], x["gv"] = (_gaussians(x.pop(k), case["degree"]) for k in ("scene", "m", "v"))
    return x


def _moments(params, seed):
    """A run some thousand steps in: Adam moments of the size of this loss's gradients."""
    r = _Draw(seed + 1)
    return {"params": params, "m": 1e-5 * r.normal(params.numel()), "v": 1e-9 * r.uniform(0.5, 2, params.numel()),
            "step": 3000}


def run(x):
    op = x["op"]
    if op == "raster":
        rgb, feat, unc, T = leg.rasterize(*x["leaves"], x["cam"], x["degree"])
        grads = torch.autograd.grad((rgb, feat, unc), x["leaves"], x["up"])
        images = [t.detach_() for t in (rgb, feat, unc)]          # kept without their graph
        return dict(zip(("rgb", "feat", "unc"), images), T=T, **{"d_" + f: g for f, g in zip(FIELDS, grads)})
    if op == "train":
        st = x["st"]
        loss = st.step(x["cam"], x["rgb"], x["target"])
        return dict(loss=loss, params=st.pv, m=st.layout.views(st.m), v=st.v)
    if op == "query":
        leg.le_preprocess(x["g"], x["cam"], x["proj"])
        img = leg.le_bin_render_fwd(x["cam"], x["proj"], x["bins"], x["img"])[3]
        p = img.unc.numel()
        rel = leg.le_query(leg.FUSED_BF16, p, x["book"], D_CLIP, x["text"], x["negs"], feat=img.feat.view(8, p),
                           dec_t=x["dec"], workspace=x["ws"], out=x["out"])
        return dict(relevancy=rel, rgb=img.rgb, feat=img.feat)
    if op == "decode":
        out = leg.le_decode(leg.FUSED_BF16, x["feat"], x["dec"], want_prob=True, workspace=x["ws"])
        return dict(argmax=out["argmax"], prob=out["prob"])
    if op == "decode_train":
        out = leg.le_decode(leg.FUSED_BF16, x["feat"], x["dec"], x["unc"], x["target"], want_argmax=False,
                            workspace=x["ws"])
        return dict(loss=out["loss"], d_feat=out["d_feat"], d_unc=out["d_unc"], dW=out["dW"])
    if op == "export":
        return leg.le_feature_map(x["feat"], x["dec"], x["book"], out=x["out"])
    if op == "quantize":
        return dict(zip(("indices", "r", "p", "loss"), leg.le_quantize(x["f"], x["book"], workspace=x["ws"])))
    if op == "quantize_grad":
        return leg.le_quantize_grad(x["f"], x["book"], x["r"], workspace=x["ws"])
    if op == "smooth":
        s = x["scene"]
        loss, d_feat, grads, _ = leg.le_smooth(s["means"], s["feat"], s["unc"], x["mlp"])
        return dict(loss=loss, d_feat=d_feat, grads=grads)
    out = leg.le_densify(x["g"], x["gm"], x["gv"], x["acc"], x["cnt"], x["noise"], max_radius=x["radius"], **DENSIFY)
    return {k: {f: getattr(o, f) for f in FIELDS} for k, o in zip("gmv", out)}


# ------------------------------------------------------------------------------------------------ work
def work(case):
    """Compulsory bytes (inputs once, outputs once) and arithmetic of one pass.  Compositing is counted at
    100 blended Gaussians a pixel (42 flops forward, 97 backward), the mean of the 1M scene."""
    op, codes = case["op"], case.get("codes", 0)
    per = 4 * (20 + 3 * (case.get("degree", 3) + 1) ** 2)                        # bytes of one Gaussian
    p = case.get("pixels") or case.get("w", 0) * case.get("h", 0)
    h = case.get("hidden", 64)
    mlp = 2 * (8 * h + 2 * h * h + 2 * h * codes)
    if op == "raster":
        return {"bytes": 2 * per * case["n"] + 4 * 25 * p, "flops": 13900 * min(p, case["n"] * 256)}
    if op == "train":
        return {"bytes": 6 * per * case["n"] + 4 * 16 * p, "flops": 13900 * min(p, case["n"] * 256) + 3 * mlp * p}
    if op == "query":
        return {"bytes": per * case["n"] + 4 * (11 + case["prompts"]) * p,
                "flops": (4200 + mlp + 2 * codes * codes) * p}
    if op == "decode":
        return {"bytes": 4 * (9 + codes) * p, "flops": mlp * p}
    if op == "decode_train":
        return {"bytes": 4 * 19 * p, "flops": 3 * mlp * p}
    if op == "export":
        return {"bytes": (4 * 8 + 2 * D) * p, "flops": (mlp + 2 * codes * D) * p}
    if op == "quantize":
        return {"bytes": (2 * D + 4) * case["features"], "flops": 2 * codes * D * case["features"]}
    if op == "quantize_grad":
        return {"bytes": 2 * D * case["features"] + 8 * codes * D, "flops": 4 * codes * D * case["features"]}
    if op == "smooth":
        return {"bytes": 4 * 20 * case["n"], "flops": 6 * (3 * 128 + 2 * 128 * 128 + 8 * 128) * case["n"]}
    return {"bytes": 6 * per * case["n"] + 12 * case["n"], "flops": 100 * case["n"]}


# ------------------------------------------------------------------------------------------------ 64 bits
def _sh(d, degree):
    """Real spherical harmonics with the Condon-Shortley sign, k = l^2 + l + m."""
    x, y, z = d.unbind(1)
    pi = math.pi
    y0 = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    c = math.sqrt(3 / (4 * pi))
    y1 = [-c * y, c * z, -c * x]
    c = math.sqrt(15 / (4 * pi))
    y2 = [c * x * y, -c * y * z, math.sqrt(5 / (16 * pi)) * (3 * z * z - 1), -c * x * z, c / 2 * (x * x - y * y)]
    a, b, c = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
    y3 = [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (5 * z * z - 1),
          math.sqrt(7 / (16 * pi)) * z * (5 * z * z - 3), -c * x * (5 * z * z - 1), b / 2 * z * (x * x - y * y),
          -a * x * (x * x - 3 * y * y)]
    return torch.stack(sum([y0, y1, y2, y3][:degree + 1], []), 1)


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)


def _project(s, cam, degree):
    """Screen mean, conic, opacity, 12 channels; and (depth, radius, extent, visible) without gradient."""
    view = torch.tensor(np.asarray(cam.view), dtype=torch.float64, device=DEV).view(3, 4)
    R, t = view[:, :3], s["means"] @ view[:, :3].t() + view[:, 3]
    M = _rotation(s["quats"]) * s["log_scales"].exp()[:, None, :]
    tz = t[:, 2]
    tz = torch.where(tz > cam.near, tz, torch.ones_like(tz))
    xn, yn = t[:, 0] / tz, t[:, 1] / tz
    xc = xn.clamp(-0.65 * cam.W / cam.fx, 0.65 * cam.W / cam.fx)
    yc = yn.clamp(-0.65 * cam.H / cam.fy, 0.65 * cam.H / cam.fy)
    J0 = torch.stack([cam.fx / tz, torch.zeros_like(tz), -cam.fx * xc / tz], 1) @ R
    J1 = torch.stack([torch.zeros_like(tz), cam.fy / tz, -cam.fy * yc / tz], 1) @ R
    A0, A1 = (J0[:, None, :] @ M)[:, 0], (J1[:, None, :] @ M)[:, 0]
    a, b, c = (A0 * A0).sum(1) + 0.3, (A0 * A1).sum(1), (A1 * A1).sum(1) + 0.3
    det = a * c - b * b
    mean = torch.stack([cam.fx * xn + cam.cx, cam.fy * yn + cam.cy], 1)
    d = s["means"] - torch.tensor(np.asarray(cam.campos), dtype=torch.float64, device=DEV)
    basis = _sh(d / d.norm(dim=1, keepdim=True), degree)
    rgb = (torch.einsum("nk,nkc->nc", basis, s["sh"]) + 0.5).clamp_min(0)
    o = torch.sigmoid(s["opacity_raw"])
    with torch.no_grad():
        mid = 0.5 * (a + c)
        radius = (3 * (mid + (mid * mid - det).clamp_min(0.1).sqrt()).sqrt()).ceil()
        reach = 2 * (255 * o).clamp_min(1e-300).log()
        extent = torch.stack([a, c], 1).mul(reach.clamp_min(0)[:, None]).sqrt() + 1e-3
        rest = t[:, 2], radius, extent, (t[:, 2] > cam.near) & (reach > -1e-3)
    return mean, torch.stack([c, -b, a], 1) / det[:, None], o, torch.cat([rgb, s["feat"], s["unc"][:, None]], 1), rest


def _lists(mean, rest, tx, ty):
    """Every tile's Gaussians in depth order: ids, and the tiles' starts."""
    depth, radius, extent, visible = rest
    size = torch.tensor([tx, ty], device=DEV)
    lo = ((mean - radius[:, None]) / 16).floor()
    hi = ((mean + radius[:, None] + 15) / 16).floor()
    lo = torch.maximum(lo, ((mean - extent - 15) / 16).ceil()).clamp_min(0)     # no pixel outside reaches 1/255
    hi = torch.minimum(torch.minimum(hi, ((mean + extent) / 16).floor() + 1), size)
    span = (hi - lo).clamp_min(0).long() * visible[:, None]
    order = torch.sort(depth.float(), stable=True)[1]
    lo, span = lo.long()[order], span[order]
    count = span[:, 0] * span[:, 1]
    gid = torch.repeat_interleave(order, count)
    at = torch.arange(len(gid), device=DEV) - torch.repeat_interleave(count.cumsum(0) - count, count)
    wide = torch.repeat_interleave(span[:, 0], count)
    tile = torch.repeat_interleave(lo[:, 1], count) + at // wide.clamp_min(1)
    tile = tile * tx + torch.repeat_interleave(lo[:, 0], count) + at % wide.clamp_min(1)
    tile, by = torch.sort(tile.int(), stable=True)
    starts = torch.searchsorted(tile, torch.arange(tx * ty + 1, device=DEV, dtype=torch.int32))
    return gid[by], starts


def _alpha(screen, ids, ok, tiles, tx):
    """Blending weights' alpha [tiles, entries, 256 pixels]."""
    mean, conic, o = screen[:3]
    pix = torch.arange(256, device=DEV)
    dx = mean[ids][..., 0, None] - ((tiles % tx * 16)[:, None] + pix % 16)[:, None, :]
    dy = mean[ids][..., 1, None] - ((tiles // tx * 16)[:, None] + pix // 16)[:, None, :]
    A, B, C = conic[ids][..., None, :].unbind(-1)
    power = -0.5 * (A * dx * dx + C * dy * dy) - B * dx * dy
    a = (o[ids][..., None] * power.clamp_max(0).exp()).clamp_max(0.99)
    return torch.where(ok[..., None] & (power <= 0) & (a >= 1 / 255), a, torch.zeros_like(a))


def _entries(gid, starts, tiles, begin, length):
    at = starts[tiles][:, None] + begin + torch.arange(length, device=DEV)
    ok = at < starts[tiles + 1][:, None]
    return gid[torch.where(ok, at, torch.zeros_like(at))] if len(gid) else at * 0, ok


def _blend(screen, gid, starts, tiles, length, tx):
    """12 channels and transmittance of the tiles' pixels."""
    ids, ok = _entries(gid, starts, tiles, 0, length)
    a = _alpha(screen, ids, ok, tiles, tx)
    step = torch.log1p(-a)
    log_t = step.cumsum(1)
    on = (log_t.detach() >= math.log(1e-4)).to(a.dtype)
    w = a * on * (log_t - step).exp()
    return torch.einsum("blp,blc->bcp", w, screen[3][ids]), (step * on).sum(1).exp()


def _render(s, cam, degree, upstream=None):
    """Images [12, H, W] and T [H, W] in 64 bits; with upstream(images) -> dL/dimages, also dL/d of every field."""
    s = {f: t.detach().double().requires_grad_(upstream is not None) for f, t in s.items()}
    with torch.set_grad_enabled(upstream is not None):
        *screen, rest = _project(s, cam, degree)
    leaves = [t.detach().requires_grad_(upstream is not None) for t in screen]
    tx, ty = cam.tiles_x, cam.tiles_y
    gid, starts = _lists(leaves[0].detach(), rest, tx, ty)
    with torch.no_grad():                                          # how deep every tile reads its list
        need = torch.zeros(tx * ty, dtype=torch.int64, device=DEV)
        log_t = torch.zeros(tx * ty, 256, dtype=torch.float64, device=DEV)
        live, begin = torch.arange(tx * ty, device=DEV), 0
        while len(live := live[(starts[live + 1] - starts[live] > begin) & (log_t[live] >= math.log(1e-4)).any(1)]):
            for part in live.split(512):
                log_t[part] += torch.log1p(-_alpha(leaves, *_entries(gid, starts, part, begin, 64), part, tx)).sum(1)
            begin += 64
            need[live] = begin
    order, groups, i = torch.sort(need)[1], [], 0
    sorted_need = need[order].tolist()
    while i < len(order):
        j = i + 1
        while j < len(order) and (j + 1 - i) * max(sorted_need[j], 1) <= 1 << 16:
            j += 1
        groups.append((order[i:j], max(sorted_need[j - 1], 1)))
        i = j
    tiled = torch.zeros(tx * ty, 13, 256, dtype=torch.float64, device=DEV)

    def image(x):
        c = x.shape[1]
        return x.view(ty, tx, c, 16, 16).permute(2, 0, 3, 1, 4).reshape(c, ty * 16, tx * 16)[:, :cam.H, :cam.W]

    with torch.no_grad():
        for tiles, length in groups:
            out, T = _blend(leaves, gid, starts, tiles, length, tx)
            tiled[tiles, :12], tiled[tiles, 12] = out, T
    img = image(tiled).contiguous()
    if upstream is None:
        return img[:12], img[12], None
    up = torch.zeros(12, ty * 16, tx * 16, dtype=torch.float64, device=DEV)
    up[:, :cam.H, :cam.W] = upstream(img[:12])
    up = up.view(12, ty, 16, tx, 16).permute(1, 3, 0, 2, 4).reshape(tx * ty, 12, 256)
    for tiles, length in groups:
        (_blend(leaves, gid, starts, tiles, length, tx)[0] * up[tiles]).sum().backward()
    torch.autograd.backward(screen, [t.grad for t in leaves])
    return img[:12], img[12], {f: t.grad for f, t in s.items()}


def _logits(feat, dec):
    """feat [n, 8]."""
    W1, b1, W2, b2, W3, b3 = dec
    return ((feat @ W1.t() + b1).relu() @ W2.t() + b2).relu() @ W3.t() + b3


def _decode_train(feat, unc, target, dec):
    """loss (L_CE, L_u), d_feat [8, n], d_unc [n], weight gradients."""
    n = feat.shape[1]
    dec = [t.detach().double().requires_grad_() for t in dec]
    loss, df, du = torch.zeros(2, dtype=torch.float64, device=DEV), [], []
    for f, u, t in zip(feat.t().split(1 << 18), unc.split(1 << 18), target.split(1 << 18)):
        f, u = f.detach().double().requires_grad_(), u.detach().double().requires_grad_()
        ce = torch.nn.functional.cross_entropy(_logits(f, dec), t.long(), reduction="none")
        lc, lu = (ce * (1 - u)).sum() / n, u.sum() / n
        (lc + lu).backward()
        loss += torch.stack([lc.detach(), lu.detach()])
        df.append(f.grad)
        du.append(u.grad)
    return loss, torch.cat(df).t(), torch.cat(du), [t.grad for t in dec]


def _rgb_loss(img, target, kind, lam=0.2):
    x, y = img.detach().double().requires_grad_(), target.double()
    l1 = (x - y).abs().mean()
    if kind == "l1":
        return l1.detach(), torch.autograd.grad(l1, x)[0]
    g = torch.exp(-torch.arange(-5, 6, dtype=torch.float64, device=DEV) ** 2 / 4.5)
    g = g / g.sum()

    def blur(t):
        t = torch.nn.functional.pad(t, (5, 5, 5, 5))
        t = sum(g[k] * t[..., k:k + img.shape[2]] for k in range(11))
        return sum(g[k] * t[:, k:k + img.shape[1]] for k in range(11))

    mx, my = blur(x), blur(y)
    vx, vy, cxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    ssim = (2 * mx * my + 1e-4) * (2 * cxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4))
    loss = (1 - lam) * l1 + lam * (1 - ssim.mean())
    return loss.detach(), torch.autograd.grad(loss, x)[0]


def _exact_train(case, seed):
    x = _inputs(case, seed)
    p, kept = case["w"] * case["h"], {}

    def upstream(img):
        kept["rgb"], d_rgb = _rgb_loss(img[:3], x["rgb"], case["rgb_loss"])
        kept["ce"], d_feat, d_unc, kept["dW"] = _decode_train(img[3:11].reshape(8, p), img[11].reshape(p),
                                                              x["target"].reshape(p), x["dec"])
        return torch.cat([d_rgb, d_feat.reshape(8, case["h"], case["w"]), d_unc.reshape(1, case["h"], case["w"])])

    grads = _render(x["scene"], x["cam"], 3, upstream)[2]
    values = {**x["scene"], **dict(zip(DEC, x["dec"]))}
    grads.update(zip(DEC, kept["dW"]))
    order, places, off = list(FIELDS[:-1]) + list(DEC) + ["unc"], {}, 0
    for k in order:
        places[k] = (off, values[k].numel())
        off = (off + values[k].numel() + 3) // 4 * 4
    start = _moments(torch.empty(off, device=DEV), seed)
    m0, v0, step = start["m"].double(), start["v"].double(), start["step"] + 1
    params, m, flat_v = {}, {}, 0.999 * v0
    for k in order:
        o, n = places[k]
        g = grads[k].reshape(-1)
        mk = 0.9 * m0[o:o + n] + 0.1 * g
        flat_v[o:o + n] += 0.001 * g * g
        den = (flat_v[o:o + n] / (1 - 0.999 ** step)).sqrt() + 1e-8
        pk = values[k].double().reshape(-1) - 1e-3 * mk / (1 - 0.9 ** step) / den
        params[k] = (pk.clamp(0, 1) if k == "unc" else pk).view(values[k].shape)
        m[k] = mk.view(values[k].shape)
    return dict(loss=torch.cat([kept["rgb"].view(1), kept["ce"]]), params=params, m=m, v=flat_v)


def _exact_quantize(case, x):
    """Cosines with the codebook's BF16 rounding; r is an input of the gradient and an output otherwise."""
    k, grad = case["features"], "r" in x
    b = x["book"].bfloat16().double()
    nb = torch.stack([b[:, :D_CLIP].norm(dim=1), b[:, D_CLIP:].norm(dim=1)])
    uc, ud = b[:, :D_CLIP] / nb[0][:, None], b[:, D_CLIP:] / nb[1][:, None]
    r, p, cos = (torch.zeros(case["codes"], dtype=torch.float64, device=DEV) for _ in range(3))
    gc, gd = torch.zeros_like(uc), torch.zeros_like(ud)
    for f in x["f"].split(1 << 17):
        f = f.double()
        fc, fd = _unit(f[:, :D_CLIP]), _unit(f[:, D_CLIP:])
        cc, cd = fc @ uc.t(), fd @ ud.t()
        dist = cc + 0.5 * cd
        best, s = dist.argmax(1), dist.softmax(1)
        if grad:
            rr = x["r"].double()
            g = 0.5 / k * s * (rr - (s @ rr)[:, None])
            g[torch.arange(len(f), device=DEV), best] -= 1 / k
            gc += g.t() @ fc - (g * cc).sum(0)[:, None] * uc
            gd += 0.5 * (g.t() @ fd - (g * cd).sum(0)[:, None] * ud)
        else:
            r += torch.bincount(best, minlength=case["codes"]) / k
            p += s.sum(0) / k
            cos[0] += (1.5 - dist.gather(1, best[:, None])).sum() / k
    if grad:
        return torch.cat([gc / nb[0][:, None], gd / nb[1][:, None]], 1)
    lb = (r * p).sum()
    return dict(indices=None, r=r, p=p, loss=torch.stack([cos[0] + 0.5 * lb, cos[0], lb]))


def _exact_smooth(x):
    s, mlp = x["scene"], [t.detach().double().requires_grad_() for t in x["mlp"]]
    n = len(s["unc"])
    loss, d_feat = torch.zeros(1, dtype=torch.float64, device=DEV), []
    for p, f, u in zip(*(s[k].double().split(1 << 18) for k in ("means", "feat", "unc"))):
        h = p
        for i in range(0, 6, 2):
            h = (h @ mlp[i].t() + mlp[i + 1]).relu()
        out = h @ mlp[6].t() + mlp[7]
        f = f.requires_grad_()
        total = ((out - f.detach()).norm(dim=1) + u.clamp_min(0.1) * (out.detach() - f).norm(dim=1)).sum() / n
        total.backward()
        loss += total.detach()
        d_feat.append(f.grad)
    return dict(loss=loss, d_feat=torch.cat(d_feat), grads=[t.grad for t in mlp])


def _exact_densify(x):
    s, c = x["scene"], DENSIFY
    f32 = lambda v: torch.tensor(np.float32(v), device=DEV)  # noqa: E731
    big = s["log_scales"].amax(1)
    pruned = s["opacity_raw"] < f32(math.log(c["min_opacity"] / (1 - c["min_opacity"])))
    pruned |= x["radius"].float() > c["max_screen_size"]
    pruned |= big > f32(math.log(c["world_frac"] * c["scene_extent"]))
    grows = (x["cnt"] > 0) & (x["acc"] >= f32(c["grad_thresh"]) * x["cnt"].float()) & ~pruned
    split = grows & (big > f32(math.log(c["percent_dense"] * c["scene_extent"])))
    kept, clone, split = (torch.nonzero(t).view(-1) for t in (~pruned & ~split, grows & ~split, split))
    src = torch.cat([kept, clone, split.repeat_interleave(2)])
    out = {"g": {f: t[src].double() for f, t in s.items()}}
    for k in "mv":
        out[k] = {f: t[src].double() for f, t in x[k].items()}
        for t in out[k].values():
            t[len(kept):] = 0
    at = len(kept) + len(clone)
    par = {f: t[split].double() for f, t in s.items()}
    child = par["log_scales"].exp()[:, None, :] * x["noise"][split].double()
    out["g"]["means"][at:] = (par["means"][:, None] + child @ _rotation(par["quats"]).transpose(1, 2)).reshape(-1, 3)
    out["g"]["log_scales"][at:] -= math.log(1.6)
    return out


def exact(case, seed):
    op = case["op"]
    if op == "train":
        return _exact_train(case, seed)
    x = _inputs(case, seed)
    if op == "raster":
        img, T, grads = _render(x["scene"], x["cam"], case["degree"], lambda _: torch.cat([
            x["up"][0], x["up"][1], x["up"][2][None]]).double())
        return dict(rgb=img[:3], feat=img[3:11], unc=img[11], T=T, **{"d_" + f: g for f, g in grads.items()})
    if op == "query":
        img = _render(x["scene"], x["cam"], 3)[0]
        dec, book = [t.double() for t in x["dec"]], x["book"][:, :D_CLIP].double()
        q, k, rel = x["text"].double(), x["negs"].double(), []
        for f in img[3:11].reshape(8, -1).t().split(1 << 18):
            phi = _unit(_logits(f, dec).softmax(1) @ book)
            rel.append(torch.sigmoid((phi @ q.t())[:, :, None] - (phi @ k.t())[:, None, :]).amin(2))
        return dict(relevancy=torch.cat(rel).t(), rgb=img[:3], feat=img[3:11])
    if op == "decode":
        dec = [t.double() for t in x["dec"]]
        prob = torch.cat([_logits(f.double(), dec).softmax(1) for f in x["feat"].t().split(1 << 18)])
        return dict(argmax=None, prob=prob.t())
    if op == "decode_train":
        loss, d_feat, d_unc, dW = _decode_train(x["feat"], x["unc"], x["target"], x["dec"])
        return dict(loss=loss, d_feat=d_feat, d_unc=d_unc, dW=dW)
    if op == "export":
        dec, book = [t.double() for t in x["dec"]], x["book"].double()
        out = torch.empty((case["pixels"], D), device=DEV)
        for i in range(0, case["pixels"], 1 << 18):
            out[i:i + (1 << 18)] = _logits(x["feat"][:, i:i + (1 << 18)].t().double(), dec).softmax(1) @ book
        return out
    if op in ("quantize", "quantize_grad"):
        return _exact_quantize(case, x)
    return _exact_smooth(x) if op == "smooth" else _exact_densify(x)
