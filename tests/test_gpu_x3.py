"""The FP32 network on the tensor cores (three-part BF16 products): against
FP64 at the edges of its 128-pixel tiles, row pairs and channel chunks, and
with infinite, NaN and overflowing inputs.

Tolerance: a layer's sums are within 2^-22 of their terms' 2-norm (measured
1.5e-7 at K = 3456, an FP32 FMA chain 1e-6); over at most 15 layers of
activations of size ~1 the logits are within 2e-5, the sigmoids within 5e-6;
the bound is four times that."""
import numpy as np
import pytest

import scenegen as sg
from helpers import renderer, set_cam

pytestmark = pytest.mark.gpu
TOL = 2e-5


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _conv(x, layer):
    import torch
    import torch.nn.functional as Fn
    w, b = (torch.from_numpy(v.astype(np.float64)) for v in layer)
    return Fn.conv2d(x, w.permute(0, 3, 1, 2), b, padding=w.shape[1] // 2)


def _unet(x, layers, levels):
    import torch
    import torch.nn.functional as Fn
    it, skip = iter(layers), []
    for l in range(levels):
        x = _conv(_conv(x, next(it)).relu(), next(it)).relu()
        if l + 1 < levels:
            skip.append(x)
            x = Fn.max_pool2d(x, 2)
    for s in reversed(skip):
        x = torch.cat([Fn.interpolate(x, scale_factor=2, mode="nearest"), s], 1)
        x = _conv(_conv(x, next(it)).relu(), next(it)).relu()
    return _conv(x, next(it)).sigmoid()


def _run(arch, layers, F, A=None, ch=(32,), cout=4, ach=(0, 0)):
    import torch
    import paper_2202_05628_gb300 as art
    H, W, C = F.shape
    sc = sg.preset("mini")
    r = renderer(sc, profile=True)
    r.set_config(profile=True)
    cam = sg.orbit_camera(sc.centroid, W, H)
    set_cam(r, 0, cam)
    r.load_shader(arch, C, list(ch), cout, art.flat_params(layers), "f32", list(ach))
    Ft = torch.from_numpy(F).cuda()
    out = torch.empty((H, W, cout), device="cuda")
    if A is None:
        r.shade(0, Ft, out, "f32")
    else:
        r.shade_with_opacity(0, Ft, torch.from_numpy(A).cuda(), out, "f32")
    r.sync_status()
    kt = r.kernel_times()
    assert kt.get("conv_x3", (0, 0))[0] == sum(w.shape[1] == 3 for w, _ in layers), kt
    return out.cpu().numpy()


def _features(rng, H, W, C):
    F = (0.5 * rng.standard_normal((H, W, C))).astype(np.float32)
    F[rng.uniform(size=(H, W)) < 0.3] = 0.0
    return F


# one row pair and tile, ragged tiles at every level, exact tiles, more row pairs than tiles
@pytest.mark.parametrize("H,W", [(8, 8), (16, 136), (40, 264), (24, 256), (264, 16)])
def test_unet(H, W):
    import torch
    import paper_2202_05628_gb300 as art
    rng = np.random.default_rng(H * 1000 + W)
    F, layers = _features(rng, H, W, 32), sg.unet_weights(3, cin=32)
    ref = _unet(torch.from_numpy(F.astype(np.float64)).permute(2, 0, 1)[None], layers, 4)[0].permute(1, 2, 0).numpy()
    got = _run(art.ART_NET_UNET, layers, F, ch=sg.UNET_CHANNELS)
    assert np.abs(got - ref).max() < TOL


def test_two_branch():
    import torch
    import paper_2202_05628_gb300 as art
    rng = np.random.default_rng(11)
    H, W = 24, 136
    F, A = _features(rng, H, W, 16), rng.uniform(0, 1, (H, W)).astype(np.float32)
    rgb, alpha = sg.two_branch_weights(2, cin=16)
    x = _unet(torch.from_numpy(F.astype(np.float64)).permute(2, 0, 1)[None], rgb, 4)
    y = _unet(torch.cat([torch.from_numpy(A.astype(np.float64))[None, None], x], 1), alpha, 2)
    ref = torch.cat([x, y], 1)[0].permute(1, 2, 0).numpy()
    got = _run(art.ART_NET_TWO_BRANCH, rgb + alpha, F, A, ch=sg.UNET_CHANNELS, ach=sg.ALPHA_CHANNELS)
    assert np.abs(got - ref).max() < TOL


@pytest.mark.parametrize("H,W,C,cout", [(1, 1, 4, 4), (3, 129, 8, 3), (5, 127, 16, 4), (131, 2, 32, 32), (7, 300, 16, 1)])
def test_tiny(H, W, C, cout):
    import torch
    import paper_2202_05628_gb300 as art
    rng = np.random.default_rng(H * 100 + W)
    F, layers = _features(rng, H, W, C), sg.tiny_net_weights(1, cin=C, cout=cout)
    x = torch.from_numpy(F.astype(np.float64)).permute(2, 0, 1)[None]
    ref = _conv(_conv(_conv(x, layers[0]).relu(), layers[1]).relu(), layers[2]).sigmoid()[0].permute(1, 2, 0).numpy()
    assert np.abs(_run(art.ART_NET_TINY, layers, F, cout=cout) - ref).max() < TOL


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3.4e38, -3.4e38, 1e-40])
def test_extreme_inputs_propagate_as_in_fp32(value):
    """One extreme input value: the outputs are not finite, saturated or
    finite where an FP32 network's are (ReLU maps NaN to 0, as fmaxf does)."""
    import torch
    import paper_2202_05628_gb300 as art
    rng = np.random.default_rng(4)
    F, layers = _features(rng, 12, 20, 16), sg.tiny_net_weights(2, cin=16)
    F[6, 9, 5] = value
    relu = lambda t: torch.where(t > 0, t, torch.zeros_like(t))
    x = torch.from_numpy(F.astype(np.float64)).permute(2, 0, 1)[None]
    big = float(np.finfo(np.float32).max)
    for k in (0, 1, 2):  # (an FP32 sum beyond the largest value is infinite)
        x = _conv(x, layers[k])
        x = torch.where(x.abs() > big, x * np.inf, x)
        x = relu(x) if k < 2 else x
    ref = x.sigmoid()[0].permute(1, 2, 0).numpy()
    got = _run(art.ART_NET_TINY, layers, F)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    ok = ~np.isnan(ref)
    assert np.abs(got[ok] - ref[ok]).max() < TOL
