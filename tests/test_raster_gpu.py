"""GPU parity of the rasterizer (preprocess, binning, render forward and
backward) against the FP64 oracle, through the C ABI.

Bars: bit-exact for integers (tiles, keys, sorted order, ranges, n_contrib);
1e-5 relative (per-tensor infinity norm) for per-Gaussian FP32 values; 1e-4
for images, T_final and all gradients.  Pixels the oracle flags as sitting on
a threshold (flip pixels) are excluded from image comparisons and get zero
upstream gradient on both sides.
"""
import numpy as np
import pytest
import torch

from paper_2311_18482_gb300 import synth
from parity import rel_err, to_np, upstream

pytestmark = pytest.mark.gpu


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def _run(leg, sc, cam):
    g = leg.Gaussians.from_scene(sc)
    proj = leg.le_preprocess(g, cam)
    ids, ranges, K, keys = leg.le_bin_sort(cam, proj, want_keys=True)
    img = leg.le_render_fwd(cam, proj, ids, ranges)
    torch.cuda.synchronize()
    return g, proj, ids, ranges, K, keys, img


def _check_preprocess(proj, sc, kp, pr):
    vis = kp["tiles"] > 0
    assert np.array_equal(to_np(proj.tiles_touched), kp["tiles"])
    assert np.array_equal(to_np(proj.radius), kp["radius"])
    assert np.array_equal(to_np(proj.rect).view(np.uint16).astype(np.int32), kp["rect"])
    assert np.array_equal(to_np(proj.depth).view(np.uint32)[vis], kp["depth"].view(np.uint32)[vis])
    assert np.array_equal(to_np(proj.tile_ellipse).view(np.uint32), kp["ell"].view(np.uint32))
    sp = to_np(proj.splat)
    assert np.array_equal(sp[vis, 0:2].view(np.uint32), kp["mean2d"][vis].view(np.uint32))
    l2e = np.log2(np.e)
    assert rel_err(sp[vis, 2:5] / np.array([l2e / 2, l2e, l2e / 2]), pr["conic"][vis]) < 1e-5   # base-2 units
    assert rel_err(sp[vis, 5], pr["opacity"][vis]) < 1e-5
    assert rel_err(sp[vis, 6:9], pr["rgb"][vis]) < 1e-5
    assert np.array_equal(sp[vis, 9], sc.unc[vis])
    assert np.array_equal(sp[vis, 10:18], sc.feat[vis])
    assert np.all(sp[~vis] == 0)


def _check_image(img, ref, mask=None):
    ok = ref["flip"] == 0
    if mask is not None:
        ok &= mask
    assert ok.mean() > 0.99
    for k, r in (("rgb", ref["rgb"]), ("feat", ref["feat"])):
        assert rel_err(to_np(getattr(img, k))[:, ok], r[:, ok]) < 1e-4, k
    assert rel_err(to_np(img.unc)[ok], ref["unc"][ok]) < 1e-4
    assert rel_err(to_np(img.T)[ok], ref["T"][ok]) < 1e-4
    assert np.array_equal(to_np(img.n_contrib)[ok], ref["n_contrib"][ok])


@pytest.mark.parametrize("case", [("c1", {}), ("c1", dict(n=700, W=100, H=75)), ("c2", dict(n=20000, W=320, H=240))])
def test_forward_parity(leg, orc, case):
    name, kw = case
    c = synth.config(name, **kw)
    sc, cam = c["scene"], c["camera"]
    cam.bg = np.array([0.1, 0.2, 0.3], np.float32)
    g, proj, ids, ranges, K, keys, img = _run(leg, sc, cam)
    ref = orc.forward(sc, cam)
    _check_preprocess(proj, sc, ref["kp"], ref["proj"])
    assert K == len(ref["vals"])
    assert np.array_equal(to_np(keys).view(np.uint64), ref["keys"])
    assert np.array_equal(to_np(ids).view(np.uint32), ref["vals"])
    assert np.array_equal(to_np(ranges).view(np.uint32), ref["ranges"])
    _check_image(img, ref["img"])


@pytest.mark.parametrize("case", [("c1", {}), ("c1", dict(n=700, W=100, H=75)), ("c2", dict(n=20000, W=320, H=240))])
def test_backward_parity(leg, orc, case):
    name, kw = case
    c = synth.config(name, **kw)
    sc, cam = c["scene"], c["camera"]
    cam.bg = np.array([0.1, 0.2, 0.3], np.float32)
    g, proj, ids, ranges, K, keys, img = _run(leg, sc, cam)
    ref = orc.forward(sc, cam)
    ok = ref["img"]["flip"] == 0
    dr, df, du = upstream(np.random.default_rng(11), cam.H, cam.W, ok)
    grads, grad2d = leg.le_render_bwd(cam, g, proj, ids, ranges, img, _t(dr), _t(df), _t(du))
    torch.cuda.synchronize()
    g2 = orc.render_bwd(cam, sc, ref["proj"], ref["vals"], ref["ranges"], dr, df, du)
    gp = orc.project_bwd(sc, cam, ref["kp"]["tiles"], g2["mean2d"], g2["conic"], g2["opacity"], g2["rgb"])
    G = to_np(grad2d)
    assert rel_err(G[:, 0:2], g2["mean2d"]) < 1e-4
    assert rel_err(G[:, 2:5], g2["conic"]) < 1e-4
    assert rel_err(G[:, 5], g2["opacity"]) < 1e-4
    assert rel_err(G[:, 6:9], g2["rgb"]) < 1e-4
    assert rel_err(G[:, 9], g2["unc"]) < 1e-4
    assert rel_err(G[:, 10:18], g2["feat"]) < 1e-4
    for k in ("means", "log_scales", "quats", "opacity_raw", "sh"):
        assert rel_err(to_np(getattr(grads, k)), gp[k]) < 1e-4, k
    assert rel_err(to_np(grads.feat), g2["feat"]) < 1e-4
    assert rel_err(to_np(grads.unc), g2["unc"]) < 1e-4


@pytest.mark.parametrize("W,H", [(16, 16), (37, 21), (608, 256), (624, 256)])
def test_backward_few_and_many_tiles(leg, orc, W, H):
    """The backward's two layouts on both sides of their line (608 tiles) and on odd list lengths, against
    the oracle's adjoint: 1e-4 of each field's largest gradient."""
    c = synth.config("c1", n=601, W=W, H=H)
    sc, cam = c["scene"], c["camera"]
    cam.bg = np.array([0.3, 0.1, 0.2], np.float32)
    ref = orc.forward(sc, cam)
    ok = ref["img"]["flip"] == 0
    dr, df, du = upstream(np.random.default_rng(W), H, W, ok)
    g, proj, ids, ranges, K, keys, img = _run(leg, sc, cam)
    grads, _ = leg.le_render_bwd(cam, g, proj, ids, ranges, img, _t(dr), _t(df), _t(du))
    g2 = orc.render_bwd(cam, sc, ref["proj"], ref["vals"], ref["ranges"], dr, df, du)
    gp = orc.project_bwd(sc, cam, ref["kp"]["tiles"], g2["mean2d"], g2["conic"], g2["opacity"], g2["rgb"])
    for k in ("means", "log_scales", "quats", "opacity_raw", "sh"):
        assert rel_err(to_np(getattr(grads, k)), gp[k]) < 1e-4, k
    assert rel_err(to_np(grads.feat), g2["feat"]) < 1e-4
    assert rel_err(to_np(grads.unc), g2["unc"]) < 1e-4


@pytest.mark.parametrize("W,H", [(384, 304), (400, 304)])
def test_backward_layouts_at_their_line(leg, orc, W, H):
    """The last image size of the two-pixel layout (456 tiles) and the first of the four-pixel one."""
    test_backward_few_and_many_tiles(leg, orc, W, H)


@pytest.mark.parametrize("W,H", [(16, 16), (512, 320)])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_backward_keeps_non_finite_channels_to_their_pixels(leg, W, H, bad):
    """Two Gaussians in one tile, no pixel blending both: the gradients of the nearer one are bit for bit the
    same whether or not a channel of the other is finite, in both layouts of the backward (1 and 640 tiles)."""
    cam = synth.look_at_camera((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), W, H, 60.0)
    cam.fx, cam.fy, cam.cx, cam.cy = 100.0, 100.0, 7.5, 7.5
    z = np.array([3.0, 4.0])                        # camera depths; pixels (12, 6) and (3, 6)
    px = np.array([12.0, 3.0])
    means = np.stack([(px - cam.cx) * z / cam.fx, (6.0 - cam.cy) * z / cam.fy, z], 1)
    R = np.asarray(cam.view, np.float64).reshape(3, 4)
    means = (means - R[:, 3]) @ R[:, :3]            # back into the world
    quats = np.tile(np.array([1.0, 0, 0, 0]), (2, 1))
    rng = np.random.default_rng(3)
    up = [_t(a) for a in upstream(rng, H, W)]
    fixed = (_t(means), _t(np.full((2, 3), -6.0)), _t(quats), _t(np.full(2, 2.0)), _t(rng.uniform(-1, 1, (2, 1, 3))))
    feat, unc = rng.standard_normal((2, 8)), _t(rng.uniform(0, 1, 2))

    def grads():
        g = leg.Gaussians(*fixed, _t(feat), unc, 0)
        proj = leg.le_preprocess(g, cam)
        ids, ranges, K, _ = leg.le_bin_sort(cam, proj)
        img = leg.le_render_fwd(cam, proj, ids, ranges)
        out, grad2d = leg.le_render_bwd(cam, g, proj, ids, ranges, img, *up)
        torch.cuda.synchronize()
        assert K == 2 and np.abs(to_np(proj.splat[:, 0]) - px).max() < 1e-2
        assert int(img.n_contrib[6, 12]) == 1 and int(img.n_contrib[6, 3]) == 2
        return {k: to_np(getattr(out, k))[0] for k in ("means", "log_scales", "quats", "opacity_raw", "sh", "feat",
                                                       "unc")}, to_np(grad2d)[0]

    want, want2d = grads()
    assert np.abs(want2d[:18]).min() > 0
    feat[1, 5] = bad
    got, got2d = grads()
    assert np.array_equal(got2d[:18], want2d[:18])
    for k, v in want.items():
        assert np.array_equal(got[k], v), k


def test_autograd_function(leg, orc):
    c = synth.config("c1", n=800, W=64, H=64)
    sc, cam = c["scene"], c["camera"]
    ref = orc.forward(sc, cam)
    ok = ref["img"]["flip"] == 0
    dr, df, du = upstream(np.random.default_rng(12), cam.H, cam.W, ok)
    params = [torch.from_numpy(getattr(sc, k)).cuda().requires_grad_(True)
              for k in ("means", "log_scales", "quats", "opacity_raw", "sh", "feat", "unc")]
    rgb, feat, unc, T = leg.rasterize(*params, cam, sc.sh_degree)
    loss = (rgb * _t(dr)).sum() + (feat * _t(df)).sum() + (unc * _t(du)).sum()
    loss.backward()
    g2 = orc.render_bwd(cam, sc, ref["proj"], ref["vals"], ref["ranges"], dr, df, du)
    gp = orc.project_bwd(sc, cam, ref["kp"]["tiles"], g2["mean2d"], g2["conic"], g2["opacity"], g2["rgb"])
    for p, k in zip(params, ("means", "log_scales", "quats", "opacity_raw", "sh")):
        assert rel_err(to_np(p.grad), gp[k]) < 1e-4, k
    assert rel_err(to_np(params[5].grad), g2["feat"]) < 1e-4
    assert rel_err(to_np(params[6].grad), g2["unc"]) < 1e-4


def test_autograd_memory_is_given_back(leg):
    """A view's buffers go once its outputs and graph are dropped, without a garbage collection; an
    output the loss leaves out gets a zero gradient."""
    c = synth.config("c1", n=800, W=64, H=64)
    params = [torch.from_numpy(getattr(c["scene"], k)).cuda().requires_grad_(True)
              for k in ("means", "log_scales", "quats", "opacity_raw", "sh", "feat", "unc")]

    def view():
        rgb = leg.rasterize(*params, c["camera"], c["scene"].sh_degree)[0]
        return torch.autograd.grad(rgb.sum(), params)

    grads = view()
    assert not grads[5].any() and not grads[6].any() and grads[4].any()
    del grads
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    for _ in range(3):
        view()
    torch.cuda.synchronize()
    assert torch.cuda.memory_allocated() == before


def test_degenerate_scenes(leg, orc):
    # all Gaussians behind the camera: K = 0, background everywhere, zero gradients
    c = synth.config("c1", n=50, W=40, H=24)
    sc, cam = c["scene"], c["camera"]
    cam.bg = np.array([0.25, 0.5, 0.75], np.float32)
    sc.means[:, 2] = -10.0
    g, proj, ids, ranges, K, keys, img = _run(leg, sc, cam)
    assert K == 0
    assert np.all(to_np(ranges) == 0)
    assert np.allclose(to_np(img.rgb), cam.bg[:, None, None])
    assert np.all(to_np(img.T) == 1) and np.all(to_np(img.n_contrib) == 0)
    dr, df, du = upstream(np.random.default_rng(0), cam.H, cam.W)
    grads, _ = leg.le_render_bwd(cam, g, proj, ids, ranges, img, _t(dr), _t(df), _t(du))
    assert torch.all(grads.means == 0) and torch.all(grads.sh == 0)
    # single Gaussian, empty scene
    c1 = synth.config("c1", n=1, W=16, H=16)
    g, proj, ids, ranges, K, keys, img = _run(leg, c1["scene"], c1["camera"])
    ref = orc.forward(c1["scene"], c1["camera"])
    assert K == len(ref["vals"])
    _check_image(img, ref["img"])
    c0 = synth.config("c1", n=0, W=16, H=16)
    g, proj, ids, ranges, K, keys, img = _run(leg, c0["scene"], c0["camera"])
    assert K == 0 and np.all(to_np(img.T) == 1)


@pytest.mark.parametrize("n", [1, 31, 33, 2047, 2049, 16384, 16385])
def test_binning_order_on_both_sorts(leg, orc, n):
    """Few Gaussians are ordered by counting, more by radix passes: with every depth shared by two or
    more Gaussians, the lists and ranges equal the oracle's stable sort."""
    c = synth.config("c1", n=n, W=64, H=48)
    sc, cam = c["scene"], c["camera"]
    sc.means[:] = sc.means[np.arange(n) // 2 % 700]
    sc.log_scales -= 1.0
    g = leg.Gaussians.from_scene(sc)
    ids, ranges, K, _ = leg.le_bin_sort(cam, leg.le_preprocess(g, cam))
    ref = orc.forward(sc, cam)
    assert K == len(ref["vals"])
    assert np.array_equal(ids.cpu().numpy().view(np.uint32), ref["vals"])
    assert np.array_equal(ranges.cpu().numpy().view(np.uint32).reshape(-1), np.asarray(ref["ranges"]).reshape(-1))


@pytest.mark.parametrize("n", [100_003, 450_000, 450_001, 1_000_003])
def test_depth_order_on_both_tiles(leg, n):
    """Both tile sizes of the radix sort: on one column of tiles, every list is in (depth, index) order."""
    rng = np.random.default_rng(n)
    c = synth.config("c1", n=4, W=16, H=16)
    cam = c["camera"]
    depth = torch.from_numpy(rng.choice(rng.uniform(0.5, 9.0, n // 3).astype(np.float32), n)).cuda()
    proj = leg.Projected.empty(n)
    proj.depth.copy_(depth)
    seen = torch.from_numpy((rng.uniform(size=n) < 0.02).astype(np.int32)).cuda()
    proj.tiles_touched.copy_(seen)
    proj.rect.copy_(torch.tensor([0, 0, 1, 1], dtype=torch.int16).cuda().expand(n, 4) * seen[:, None].to(torch.int16))
    # an ellipse that reaches the whole tile: centred on it, a long way wide and high
    proj.tile_ellipse.copy_(torch.tensor([8.0, 8.0, 0.0, 1.0, 1e6, 0.0, 0.25, 0.25]).cuda().expand(n, 8))
    ids, ranges, K, _ = leg.le_bin_sort(cam, proj)
    idx = torch.nonzero(seen).view(-1)
    order = torch.sort(depth[idx], stable=True)[1]
    assert K == len(idx)
    assert torch.equal(ids.long(), idx[order])


def test_deterministic_binning(leg):
    c = synth.config("c2", n=50000, W=320, H=240)
    sc, cam = c["scene"], c["camera"]
    a = _run(leg, sc, cam)
    b = _run(leg, sc, cam)
    assert torch.equal(a[2], b[2]) and torch.equal(a[3], b[3])
    assert torch.equal(a[6].rgb, b[6].rgb)


@pytest.mark.parametrize("name,lazy", [("c3", False), ("c5", True)])
def test_full_size_crop_parity(leg, orc, name, lazy):
    """Full-size scenes (1M Gaussians, 1296x840): preprocess on every Gaussian,
    binning on sampled tiles, images and gradients on the 64x64 centre crop
    (upstream gradient zero elsewhere).  c3 through le_bin_sort + le_render_fwd;
    c5 (the training step's view) through le_bin_render_fwd, the lazily placed
    lists the training step renders from, whose tiles hold only the entries
    some pixel reads: those are compared with the oracle's list prefix."""
    c = synth.config(name)
    sc, cam = c["scene"], c["camera"]
    if lazy:
        g = leg.Gaussians.from_scene(sc)
        proj = leg.le_preprocess(g, cam)
        ids, ranges, K, img = leg.le_bin_render_fwd(cam, proj)
        torch.cuda.synchronize()
    else:
        g, proj, ids, ranges, K, keys, img = _run(leg, sc, cam)
    kp = orc.keypath(sc, cam)
    pr = orc.project(sc, cam, kp["tiles"])
    _check_preprocess(proj, sc, kp, pr)
    assert K == orc.bin_count(kp) < int(kp["tiles"].astype(np.int64).sum())
    ids_np = to_np(ids).view(np.uint32)
    rg = to_np(ranges).view(np.uint32)
    nc = to_np(img.n_contrib) & ((1 << 30) - 1)
    rng = np.random.default_rng(3)
    for t in rng.choice(cam.tiles_x * cam.tiles_y, 12, replace=False):
        tx, ty = t % cam.tiles_x, t // cam.tiles_x
        want = orc.tile_list(kp, tx, ty)
        assert rg[t, 1] - rg[t, 0] == len(want)
        m = int(nc[ty * 16:(ty + 1) * 16, tx * 16:(tx + 1) * 16].max()) if lazy else len(want)
        assert np.array_equal(ids_np[rg[t, 0]:rg[t, 0] + m], want[:m])
    x0, y0 = (cam.W // 2 - 32) // 16 * 16, (cam.H // 2 - 32) // 16 * 16
    win = (x0, y0, x0 + 64, y0 + 64)
    tl = [(tx, ty) for ty in range(y0 // 16, y0 // 16 + 4) for tx in range(x0 // 16, x0 // 16 + 4)]
    vals, rr = orc.lists_for_tiles(cam, kp, tl)
    ref = orc.render(cam, sc, pr, vals, rr, win)
    sub = lambda a: a[..., y0:y0 + 64, x0:x0 + 64]
    ok = ref["flip"] == 0
    for k in ("rgb", "feat"):
        assert rel_err(sub(to_np(getattr(img, k)))[:, ok], ref[k][:, ok]) < 1e-4, k
    assert rel_err(sub(to_np(img.T))[ok], ref["T"][ok]) < 1e-4
    assert np.array_equal(sub(to_np(img.n_contrib))[ok], ref["n_contrib"][ok])
    dr, df, du = upstream(np.random.default_rng(4), 64, 64, ok)
    DR, DF, DU = np.zeros((3, cam.H, cam.W)), np.zeros((8, cam.H, cam.W)), np.zeros((cam.H, cam.W))
    DR[:, y0:y0 + 64, x0:x0 + 64], DF[:, y0:y0 + 64, x0:x0 + 64], DU[y0:y0 + 64, x0:x0 + 64] = dr, df, du
    grads, grad2d = leg.le_render_bwd(cam, g, proj, ids, ranges, img, _t(DR), _t(DF), _t(DU))
    torch.cuda.synchronize()
    g2 = orc.render_bwd(cam, sc, pr, vals, rr, dr, df, du, window=win)
    gp = orc.project_bwd(sc, cam, kp["tiles"], g2["mean2d"], g2["conic"], g2["opacity"], g2["rgb"])
    for k in ("means", "log_scales", "quats", "opacity_raw", "sh"):
        assert rel_err(to_np(getattr(grads, k)), gp[k]) < 1e-4, k
    assert rel_err(to_np(grads.feat), g2["feat"]) < 1e-4
    assert rel_err(to_np(grads.unc), g2["unc"]) < 1e-4


def test_c4_query_render_crop(leg, orc):
    """The query-render workload (3M Gaussians, 1920x1080, 256 codes x 896 dims): render, then the fused BF16
    decode and relevancy on the whole view; the FP64 oracle renders the 128x128 centre crop from brute-force
    tile lists, decodes it and forms the relevancy.  Pixels on an alpha threshold are excluded."""
    import paper_2311_18482_gb300 as L
    c = synth.config("c4")
    sc, cam, dec, qin = c["scene"], c["camera"], c["decoder"], c["query"]
    g, proj, ids, ranges, K, keys, img = _run(leg, sc, cam)
    P = cam.W * cam.H
    dec_t = tuple(_t(getattr(dec, k)) for k in ("W1", "b1", "W2", "b2", "W3", "b3"))
    rel = L.le_query(L.FUSED_BF16, P, _t(qin.codebook), qin.d_clip, _t(qin.text), _t(qin.negs), feat=img.feat,
                     dec_t=dec_t)
    L.le_device_status()
    kp = orc.keypath(sc, cam)
    assert K == orc.bin_count(kp)
    pr = orc.project(sc, cam, kp["tiles"])
    x0, y0 = (cam.W // 2 - 64) // 16 * 16, (cam.H // 2 - 64) // 16 * 16
    win = (x0, y0, x0 + 128, y0 + 128)
    tl = [(tx, ty) for ty in range(y0 // 16, y0 // 16 + 8) for tx in range(x0 // 16, x0 // 16 + 8)]
    vals, rr = orc.lists_for_tiles(cam, kp, tl)
    ref = orc.render(cam, sc, pr, vals, rr, win)
    ok = (ref["flip"] == 0).ravel()
    assert ok.mean() > 0.95            # 98.7 % here: ~35k Gaussians per crop tile, K = 192.6M copies
    sub = lambda a: a[..., y0:y0 + 128, x0:x0 + 128].reshape(a.shape[0], -1)
    assert rel_err(sub(to_np(img.feat))[:, ok], ref["feat"].reshape(8, -1)[:, ok]) < 1e-4
    prob, _ = orc.softmax_argmax(orc.decoder_fwd(ref["feat"].reshape(8, -1)[:, ok], dec))
    want = orc.query(prob, qin)
    got = sub(to_np(rel).reshape(-1, cam.H, cam.W))[:, ok]
    err = float(np.max(np.abs(got - want)))
    print(f"c4 query render, {int(ok.sum())} crop pixels: max|drel| {err:.2e}, K = {K}")
    assert err <= 1e-2


def test_l1_and_adam(leg, orc):
    rng = np.random.default_rng(13)
    n = 1003
    img, tgt = rng.uniform(0, 1, n), rng.uniform(0, 1, n).astype(np.float32)
    loss = torch.zeros(1, device="cuda")
    grad = torch.empty(n, device="cuda")
    leg.le_rgb_l1(_t(img), _t(tgt), loss, grad)
    l_ref, g_ref = orc.l1(img.astype(np.float32).astype(np.float64), tgt)
    assert abs(loss.item() - l_ref) < 1e-5 * l_ref
    assert rel_err(to_np(grad), g_ref) < 1e-6
    p = rng.standard_normal(n)
    p_t, m_t, v_t = _t(p), torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda")
    p_o, m_o, v_o = p.astype(np.float32).astype(np.float64), np.zeros(n), np.zeros(n)
    for step in range(1, 4):
        gg = rng.standard_normal(n)
        leg.le_adam(p_t, _t(gg), m_t, v_t, step)
        orc.adam(p_o, gg.astype(np.float32).astype(np.float64), m_o, v_o, step)
    assert rel_err(to_np(p_t), p_o) < 1e-5
    # clamp to [0, 1] (the uncertainty's range)
    u = _t(rng.uniform(-0.5, 1.5, 64))
    leg.le_adam(u, torch.zeros(64, device="cuda"), torch.zeros(64, device="cuda"), torch.zeros(64, device="cuda"),
                1, clamp_lo=0.0, clamp_hi=1.0)
    assert float(u.min()) >= 0 and float(u.max()) <= 1


@pytest.mark.parametrize("case", [("c1", {}), ("c2", dict(n=20000, W=320, H=240)), ("c5", {}),
                                  ("c5", dict(pose=5))])
def test_lazy_bin_render_equals_full(leg, case):
    """le_bin_render_fwd (lists placed lazily, in depth phases) against
    le_bin_sort + le_render_fwd: images, T, n_contrib, K and ranges bit for
    bit; the list entries any pixel reads identical; and the backward from the
    lazy lists equal to the backward from the full lists."""
    name, kw = case
    c = synth.config(name, **kw)
    sc, cam = c["scene"], c["camera"]
    cam.bg = np.array([0.1, 0.2, 0.3], np.float32)
    g = leg.Gaussians.from_scene(sc)
    proj = leg.le_preprocess(g, cam)
    ids_f, ranges_f, K_f, _ = leg.le_bin_sort(cam, proj)
    img_f = leg.le_render_fwd(cam, proj, ids_f, ranges_f)
    ids_f, ranges_f = ids_f.clone(), ranges_f.clone()
    ids_l, ranges_l, K_l, img_l = leg.le_bin_render_fwd(cam, proj)
    torch.cuda.synchronize()
    assert K_l == K_f and torch.equal(ranges_l, ranges_f)
    for k in ("rgb", "feat", "unc", "T", "n_contrib"):
        assert torch.equal(getattr(img_l, k), getattr(img_f, k)), k
    # every entry a pixel of the tile reads is written, and equal
    nc = to_np(img_f.n_contrib)
    rg = to_np(ranges_f).view(np.uint32)
    a, b = to_np(ids_f).view(np.uint32), to_np(ids_l).view(np.uint32)
    TX = cam.tiles_x
    used = 0
    for t in range(rg.shape[0]):
        s0, e0 = rg[t]
        if e0 <= s0:
            continue
        ty, tx = divmod(t, TX)
        m = int(nc[ty * 16:(ty + 1) * 16, tx * 16:(tx + 1) * 16].max())
        assert np.array_equal(a[s0:s0 + m], b[s0:s0 + m]), t
        used += m
    print(f"{name} {kw}: K {K_f}, entries read {used} ({used / max(K_f, 1):.4f})")
    H, W = cam.H, cam.W
    dr, df, du = upstream(np.random.default_rng(2), H, W)
    gf, g2f = leg.le_render_bwd(cam, g, proj, ids_f, ranges_f, img_f, _t(dr), _t(df), _t(du))
    gl, g2l = leg.le_render_bwd(cam, g, proj, ids_l, ranges_l, img_l, _t(dr), _t(df), _t(du))
    torch.cuda.synchronize()
    # the same entries in the same order; only the order of the gradient atomics differs
    assert rel_err(to_np(g2l), to_np(g2f)) < 1e-4
    for k in ("means", "log_scales", "quats", "opacity_raw", "sh", "feat", "unc"):
        assert rel_err(to_np(getattr(gl, k)), to_np(getattr(gf, k))) < 1e-4, k


def test_lazy_capacity_retry(leg):
    """le_bin_render_fwd with room for only half of the K copies: the first call stops with
    LE_ERR_CAPACITY (K is reported, nothing is placed), and the binding's retry with room for K gives
    the lists and images of a call that had room from the start, bit for bit."""
    c = synth.config("c2", n=20000, W=320, H=240)
    sc, cam = c["scene"], c["camera"]
    g = leg.Gaussians.from_scene(sc)
    proj = leg.le_preprocess(g, cam)
    ids0, r0, K0, img0 = leg.le_bin_render_fwd(cam, proj)
    torch.cuda.synchronize()
    ref = {k: getattr(img0, k).clone() for k in ("rgb", "feat", "unc", "T", "n_contrib")}
    r0 = r0.clone()
    assert K0 > 2
    small = leg.BinSortBuffers()
    ids1, r1, K1, img1 = leg.le_bin_render_fwd(cam, proj, buffers=small, k_cap=K0 // 2)
    torch.cuda.synchronize()
    leg.le_device_status()
    assert K1 == K0 and small.k_cap >= K0 and torch.equal(r1, r0)
    for k, v in ref.items():
        assert torch.equal(getattr(img1, k), v), k
