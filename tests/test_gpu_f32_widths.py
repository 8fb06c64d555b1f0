"""FP32 networks by their widths, against FP64: those that the tensor-core
kernel refuses run on the CUDA cores (register-blocked kernel: channel counts
in fours; the other one: any), those it takes beyond the default widths run on
it, and infinite or NaN features pass through a U-Net as through any FP32 one.

Tolerances: on the CUDA cores a layer's sum is an FMA chain of up to 1152 (here)
terms, within 5e-7 of their 2-norm, under 15 layers of activations of size ~1:
1e-5 on the logits; the bound is that of the library's other FP32 tests, 1e-4.
On the tensor cores 2^-22 a layer, 2e-5 as at the default widths."""
import numpy as np
import pytest

import scenegen as sg
from helpers import renderer, set_cam
from test_gpu_x3 import TOL as TOL_X3
from test_gpu_x3 import _conv, _features, _unet

pytestmark = pytest.mark.gpu
TOL_SIMT = 1e-4


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _nchw(F):
    import torch
    return torch.from_numpy(F.astype(np.float64)).permute(2, 0, 1)[None]


def _hwc(t):
    return t[0].permute(1, 2, 0).numpy()


def _tiny(F, layers):
    x = _nchw(F)
    return _hwc(_conv(_conv(_conv(x, layers[0]).relu(), layers[1]).relu(), layers[2]).sigmoid())


def _run(arch, layers, F, A=None, ch=(32,), cout=4, ach=(0, 0), kernel="conv_x3"):
    import torch
    import paper_2202_05628_gb300 as art
    H, W, C = F.shape
    sc = sg.preset("mini")
    r = renderer(sc, profile=True)
    set_cam(r, 0, sg.orbit_camera(sc.centroid, W, H))
    r.load_shader(arch, C, list(ch), cout, art.flat_params(layers), "f32", list(ach))
    Ft = torch.from_numpy(F).cuda()
    out = torch.full((H, W, cout), -1.0, device="cuda")
    if A is None:
        r.shade(0, Ft, out, "f32")
    else:
        r.shade_with_opacity(0, Ft, torch.from_numpy(A).cuda(), out, "f32")
    r.sync_status()
    kt = r.kernel_times()
    n3 = sum(w.shape[1] == 3 for w, _ in layers)
    want = {"conv_x3": n3, "conv_simt": 0} if kernel == "conv_x3" else {"conv_x3": 0, "conv_simt": len(layers)}
    assert {k: kt.get(k, (0, 0))[0] for k in want} == want, kt
    return out.cpu().numpy()


# first level 16; a level neither 32 nor a multiple of 64; channel counts not in fours; more outputs than the fused
# head has; each with ragged rows of the kernels' 64-, 128- and 256-pixel tiles
@pytest.mark.parametrize("ch,cin,cout,H,W", [((16, 32, 48, 64), 16, 4, 16, 264), ((32, 64, 96, 128), 32, 4, 40, 136),
                                             ((13, 18, 21, 30), 7, 3, 24, 72), (sg.UNET_CHANNELS, 4, 7, 16, 72)])
def test_unet_on_cuda_cores(ch, cin, cout, H, W):
    import paper_2202_05628_gb300 as art
    F, layers = _features(np.random.default_rng(sum(ch)), H, W, cin), sg.unet_weights(3, cin, ch, cout)
    got = _run(art.ART_NET_UNET, layers, F, ch=ch, cout=cout, kernel="conv_simt")
    assert np.abs(got - _hwc(_unet(_nchw(F), layers, 4))).max() < TOL_SIMT


@pytest.mark.parametrize("mid,cin,cout,H,W", [(16, 16, 4, 5, 131), (15, 3, 4, 7, 65), (32, 8, 33, 3, 70), (64, 32, 4, 9, 129)])
def test_three_layers_on_cuda_cores(mid, cin, cout, H, W):
    import paper_2202_05628_gb300 as art
    F, layers = _features(np.random.default_rng(mid), H, W, cin), sg.tiny_net_weights(1, cin, mid, cout)
    got = _run(art.ART_NET_TINY, layers, F, ch=(mid,), cout=cout, kernel="conv_simt")
    assert np.abs(got - _tiny(F, layers)).max() < TOL_SIMT


@pytest.mark.parametrize("ch,ach,kernel", [(sg.UNET_CHANNELS, (16, 32), "conv_simt"), ((16, 32, 48, 64), (10, 22), "conv_simt"),
                                           ((32, 32, 64, 64), (32, 32), "conv_x3")])
def test_two_branches(ch, ach, kernel):
    import torch
    import paper_2202_05628_gb300 as art
    rng = np.random.default_rng(sum(ach))
    H, W = 24, 72
    F, A = _features(rng, H, W, 16), rng.uniform(0, 1, (H, W)).astype(np.float32)
    rgb, alpha = sg.two_branch_weights(2, 16, ch, ach)
    x = _unet(_nchw(F), rgb, 4)
    y = _unet(torch.cat([_nchw(A[..., None]), x], 1), alpha, 2)
    got = _run(art.ART_NET_TWO_BRANCH, rgb + alpha, F, A, ch=ch, ach=ach, kernel=kernel)
    assert np.abs(got - _hwc(torch.cat([x, y], 1))).max() < (TOL_X3 if kernel == "conv_x3" else TOL_SIMT)


@pytest.mark.parametrize("ch,cin,cout,H,W", [((32, 32, 64, 64), 32, 4, 24, 136), ((32, 64, 192, 128), 48, 1, 16, 264),
                                             ((32, 32, 32, 32), 100, 2, 8, 72), ((32, 64, 128, 512), 4, 3, 40, 24)])
def test_unet_widths_on_tensor_cores(ch, cin, cout, H, W):
    import paper_2202_05628_gb300 as art
    F, layers = _features(np.random.default_rng(sum(ch)), H, W, cin), sg.unet_weights(3, cin, ch, cout)
    got = _run(art.ART_NET_UNET, layers, F, ch=ch, cout=cout)
    assert np.abs(got - _hwc(_unet(_nchw(F), layers, 4))).max() < TOL_X3


@pytest.mark.parametrize("cin", [33, 64, 256])
def test_three_layers_with_wide_inputs_on_tensor_cores(cin):
    import paper_2202_05628_gb300 as art
    F, layers = _features(np.random.default_rng(cin), 5, 130, cin), sg.tiny_net_weights(1, cin)
    assert np.abs(_run(art.ART_NET_TINY, layers, F) - _tiny(F, layers)).max() < TOL_X3


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("x", [5, 255])
@pytest.mark.parametrize("positive", [False, True])
def test_extreme_features_pass_through_a_unet(value, x, positive):
    """One such feature, and a part of the image outside its reach.  Weights
    of both signs make it NaN, hence 0 after a ReLU; with positive ones an
    infinity reaches every level (pooled, x-phase split and sub-pixel
    tensors)."""
    import torch
    import torch.nn.functional as Fn
    import paper_2202_05628_gb300 as art
    H, W = 24, 520
    F, layers = _features(np.random.default_rng(4), H, W, 32), sg.unet_weights(3)
    if positive:  # (a layer's outputs of the size of its inputs)
        layers = [(np.abs(w) / np.abs(w).sum((1, 2, 3), keepdims=True) if w.shape[1] == 3 else w, b) for w, b in layers]
    F[9, x, 5] = value
    relu = lambda t: torch.where(t > 0, t, torch.zeros_like(t))  # (NaN to 0, as fmaxf does)
    it, t, skip = iter(layers), _nchw(F), []
    for l in range(4):
        t = relu(_conv(relu(_conv(t, next(it))), next(it)))
        if l < 3:
            skip.append(t)
            t = Fn.max_pool2d(t, 2)
    for s in reversed(skip):
        t = torch.cat([Fn.interpolate(t, scale_factor=2, mode="nearest"), s], 1)
        t = relu(_conv(relu(_conv(t, next(it))), next(it)))
    ref = _hwc(_conv(t, next(it)).sigmoid())
    ok = ~np.isnan(ref)
    assert ok.any() and ok.all() == (not positive or value != np.inf)
    got = _run(art.ART_NET_UNET, layers, F, ch=sg.UNET_CHANNELS)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.abs(got[ok] - ref[ok]).max() < TOL_X3
