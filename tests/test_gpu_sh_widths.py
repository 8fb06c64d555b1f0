"""View-dependent features against the FP64 oracle at every channel count
(32 / C hits per step of the walk) and degree, and where a pixel's reorder
buffer fills up, so that single lanes add their hits."""
import numpy as np
import pytest

import oracle
import scenegen as sg
from helpers import order_ambiguous, renderer, set_cam, set_pose

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _check(sc, pose, cam, L, coef):
    """Within 1e-4 of the oracle where rounding cannot decide the hits' order;
    returns the oracle's hits."""
    import torch
    oc = sc.octree
    A_or = oracle.pose_transforms(sc, pose)[1]
    p = oracle.render(oc, A_or, cam, hits=True)
    good = ~order_ambiguous(p, oc, cam.H, cam.W, effect=0.0)
    assert good.mean() > 0.8, good.mean()
    r = renderer(sc)
    set_pose(r, pose)
    set_cam(r, 0, cam)
    r.load_sh_features(L, coef)
    F = torch.empty((cam.H, cam.W, oc.C), device="cuda")
    A = torch.empty((cam.H, cam.W), device="cuda")
    r.render_feature_maps(0, F, A)
    assert r.sync_status()["overflow_order"] == 0
    o = oracle.render_sh(oc, A_or, cam, L, coef.astype(np.float64))
    np.testing.assert_allclose(A.cpu().numpy()[good], o["A"][good], atol=1e-4)
    np.testing.assert_allclose(F.cpu().numpy()[good], o["F"][good], atol=1e-4)
    return p


@pytest.mark.parametrize("C", [4, 8, 16, 32])
@pytest.mark.parametrize("L", [0, 1, 2, 3])
def test_sh_features_match_oracle(C, L):
    sc = sg.preset("tiny", C=C)
    oc = sc.octree
    cam = sg.orbit_camera(sc.centroid, 96, 64, az_deg=70.0 * L, fov_deg=12.0)
    coef = (0.3 * np.random.default_rng(10 * C + L).standard_normal((oc.n, (L + 1) ** 2, C))).astype(np.float32)
    p = _check(sc, sg.random_pose(3 + L), cam, L, coef)
    assert (p["nhit"] > 0).sum() > 500


@pytest.mark.parametrize("C", [4, 8, 16, 32])
def test_full_reorder_buffers(C):
    """A row of 30 voxels along the view, all within one staged chunk: a ray
    meets more of them than the 16 it can hold back, so the later ones make it
    release earlier hits one at a time."""
    rng = np.random.default_rng(C)
    n, L = 30, 2
    ijk = np.stack([np.full(n, 16), np.full(n, 16), np.arange(n)], 1).astype(np.uint16)
    w = np.zeros((n, 4), np.float32)
    w[:, 0] = 1.0
    oc = sg.Octree(5, np.array([-0.5, -0.5, -0.5], np.float32), 1.0, ijk, np.zeros((n, 4), np.uint8), w,
                   rng.standard_normal((n, C)).astype(np.float32), rng.uniform(1.0, 4.0, n).astype(np.float32),
                   np.zeros(n, np.float32))
    sc = sg.Scene(oc, sg.Skeleton(np.array([-1], np.int32), np.zeros((1, 3), np.float32)), np.zeros(3), 1.0, None, None)
    c = oc.centers().astype(np.float64)
    cam = sg.Camera(24, 20, 700.0, 700.0, 12.0, 10.0, sg.look_at(c[0] + np.array([0.002, 0.003, -2.0]), c[0]), 0.5, 4.0)
    coef = rng.standard_normal((n, (L + 1) ** 2, C)).astype(np.float32)
    p = _check(sc, sg.rest_pose(1), cam, L, coef)
    assert p["nused"].max() > 20
