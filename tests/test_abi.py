"""The C-ABI library builds, loads and exports every entry point include/leg.h
declares; argument validation answers without touching a GPU."""
import ctypes as C
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2311_18482_gb300 import build
    path = build.build()
    return C.CDLL(path)


def _declared():
    text = open(os.path.join(ROOT, "include", "leg.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(le_[a-z0-9_]+)\s*\(", text)))


def test_header_symbols_exported(lib):
    names = _declared()
    assert len(names) >= 10
    missing = [n for n in names if not hasattr(lib, n)]
    assert not missing, missing


def test_binding_covers_header():
    from paper_2311_18482_gb300 import binding
    assert set(_declared()) <= set(binding.exported_symbols())


def test_invalid_arguments_rejected_on_host(lib):
    from paper_2311_18482_gb300 import binding as b
    lib.le_last_error.restype = C.c_char_p
    ws = C.c_size_t()
    assert lib.le_bin_sort_workspace(C.c_int32(-1), C.c_int64(10), C.byref(ws)) == b.LE_ERR_INVALID_ARG
    assert lib.le_bin_sort_workspace(C.c_int32(1000), C.c_int64(1 << 33), C.byref(ws)) == b.LE_ERR_INVALID_ARG
    assert lib.le_bin_sort_workspace(C.c_int32(1000), C.c_int64(20000), C.byref(ws)) == b.LE_OK
    assert ws.value >= 2 * 8 * 1000          # two depth-sort buffers of n keys at least
    # null gaussians / camera
    assert lib.le_preprocess(None, None, None, None) == b.LE_ERR_INVALID_ARG
    assert b"null" in lib.le_last_error()
    cam = b.LeCamera()
    cam.width, cam.height, cam.fx, cam.fy = 0, 10, 1.0, 1.0
    g = b.LeGaussians()
    g.n, g.sh_degree = 0, 0
    p = b.LeProjected()
    assert lib.le_preprocess(C.byref(g), C.byref(cam), C.byref(p), None) == b.LE_ERR_INVALID_ARG
    cam.width = 10
    g.sh_degree = 4
    assert lib.le_preprocess(C.byref(g), C.byref(cam), C.byref(p), None) == b.LE_ERR_INVALID_ARG
    # fused backward + Adam: null camera / config rejected before any GPU work
    assert lib.le_render_bwd_adam(None, None, None, None, None, None, None, None, None, None, None, None, None,
                                  None, None) == b.LE_ERR_INVALID_ARG
    # the projection Adam with an extra range: negative size, unaligned extra pointer
    cam.width, cam.height = 16, 16
    g.n, g.sh_degree = 0, 0
    cfg = b.LeAdamConfig(1, 1e-3, 0.9, 0.999, 1e-8)
    f = lib.le_project_bwd_adam_extra
    args = (C.byref(cam), C.byref(g), C.byref(p), None, None, None, C.byref(cfg))
    assert f(*args, C.c_void_p(16), C.c_void_p(16), C.c_void_p(32), C.c_void_p(48), C.c_int64(-1),
             None) == b.LE_ERR_INVALID_ARG
    assert f(*args, C.c_void_p(18), C.c_void_p(16), C.c_void_p(32), C.c_void_p(48), C.c_int64(8),
             None) == b.LE_ERR_INVALID_ARG
    assert b"aligned" in lib.le_last_error()
    assert f(*args, None, None, None, None, C.c_int64(0), None) == b.LE_OK      # nothing to do
    # misaligned Adam buffers
    assert lib.le_adam(C.c_int64(8), C.c_void_p(3), C.c_void_p(16), C.c_void_p(32), C.c_void_p(48), 1,
                       C.c_float(1e-3), C.c_float(0.9), C.c_float(0.999), C.c_float(1e-8), C.c_float(0),
                       C.c_float(1), None) == b.LE_ERR_INVALID_ARG
    assert lib.le_adam(C.c_int64(8), C.c_void_p(16), C.c_void_p(16), C.c_void_p(32), C.c_void_p(48), 0,
                       C.c_float(1e-3), C.c_float(0.9), C.c_float(0.999), C.c_float(1e-8), C.c_float(0),
                       C.c_float(1), None) == b.LE_ERR_INVALID_ARG


def test_misaligned_workspaces_rejected_on_host(lib):
    """A workspace that starts off the boundary its kernels' accesses need is refused before any launch."""
    from paper_2311_18482_gb300 import binding as b
    lib.le_last_error.restype = C.c_char_p
    V, i, f, n = C.c_void_p, C.c_int32, C.c_float, C.c_size_t
    p, big = V(256), n(1 << 30)

    def refused(status):
        assert status == b.LE_ERR_INVALID_ARG and b"aligned" in lib.le_last_error()

    dec = b.LeDecoder()
    dec.d_in, dec.h1, dec.h2, dec.n_cb = 8, 64, 128, 64
    for k in ("W1", "b1", "W2", "b2", "W3", "b3"):
        setattr(dec, k, 256)
    for mode, at in ((b.FUSED_BF16, 264), (b.FUSED_BF16, 257), (b.UNFUSED_FP32, 258)):
        refused(lib.le_query(i(mode), i(100), p, C.byref(dec), p, p, i(64), i(64), p, i(1), p, i(1), p, V(at), big,
                             None))
    refused(lib.le_rgb_loss(i(16), i(16), p, p, f(0.2), p, p, V(258), big, None))
    g = b.LeGaussians(10, 0, *[256] * 7)
    o = b.LeGaussianGrads(*[256] * 7)
    cfg, out = b.LeDensifyConfig(0.1, 0.1, 1.0, 0.1, 0.0, 0.0), C.c_int64()
    refused(lib.le_densify(C.byref(cfg), C.byref(g), C.byref(o), C.byref(o), p, p, None, p, C.c_int64(20), C.byref(o),
                           C.byref(o), C.byref(o), C.byref(out), V(260), big, None))


def test_camera_takes_any_float_like_values():
    """Lists, arrays, one-column tensors and iterators give the same camera; a wrong count is refused."""
    import numpy as np
    import torch
    from types import SimpleNamespace
    from paper_2311_18482_gb300 import binding as b
    view, campos, bg = np.arange(12) / 7, np.array([1.5, -2, 3]), np.array([0.25, 0.5, 1])

    def camera(f, view=view):
        return bytes(b.camera_struct(SimpleNamespace(view=f(view), campos=f(campos), bg=f(bg), fx=1.0, fy=2, cx=3.5,
                                                     cy=4, W=16, H=8, near=0.2)))

    want = camera(lambda a: a)
    for form in (list, iter, tuple, lambda a: a.astype(np.float32), lambda a: map(float, a), torch.tensor,
                 lambda a: torch.tensor(a)[:, None], lambda a: [np.float32(v) for v in a],
                 lambda a: (v for v in a.tolist())):
        assert camera(form) == want
    for n in (11, 13):
        with pytest.raises((TypeError, ValueError)):
            camera(list, view=np.ones(n))


def test_gradients_beyond_the_parameters_are_zero(monkeypatch):
    """Gradient tensors come uninitialised where a backward writes every element; what a tensor holds past the
    rows of n and sh_degree, which no call writes, starts as zeros."""
    import torch
    from paper_2311_18482_gb300 import binding as b
    monkeypatch.setattr(torch, "empty_like", lambda t: torch.full_like(t, float("nan")))
    n, nan = 5, lambda t: bool(torch.isnan(t).all())
    make = lambda sh, feat: b.Gaussians(torch.ones(n, 3), torch.ones(n, 3), torch.ones(n, 4), torch.ones(n), sh, feat,
                                        torch.ones(n), 1).empty_like()
    exact = make(torch.ones(n, 4, 3), torch.ones(n, 8))
    assert all(nan(getattr(exact, k)) for k in ("means", "log_scales", "quats", "opacity_raw", "sh", "feat", "unc"))
    wide = make(torch.ones(n, 16, 3), torch.ones(n, 9))
    assert not wide.sh.any() and not wide.feat.any() and wide.sh.shape == (n, 16, 3) and nan(wide.means)
