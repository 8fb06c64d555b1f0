"""A device allocation that fails inside a call: the call reports it, and the
next calls neither use what is missing nor forget to allocate it again.  The
library is linked with a cudaMalloc that fails when told to."""
import numpy as np
import pytest

import scenegen as sg
import variants
from helpers import render_maps, renderer, set_cam, set_pose

pytestmark = pytest.mark.gpu
OOM, STATE = 3, 5

FAILING_MALLOC = """
#include <stddef.h>
int __real_cudaMalloc(void** p, size_t n);
static int left = -1;  /* allocations until the one that fails (negative: none) */
void fail_after(int n) { left = n; }
int pending(void) { return left >= 0; }
int __wrap_cudaMalloc(void** p, size_t n) {
  if (left >= 0 && left-- == 0) n = (size_t)1 << 60; /* more than any device has: cudaErrorMemoryAllocation */
  return __real_cudaMalloc(p, n);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return variants.library(tmp_path_factory.mktemp("alloc") / "liballoc.so", wrap=["cudaMalloc"], source=FAILING_MALLOC)


@pytest.fixture
def art(lib, monkeypatch):
    import paper_2202_05628_gb300 as art
    monkeypatch.setattr(art, "_lib", lib)
    yield art
    lib.fail_after(-1)


def _each_failure(art, lib, call):
    """call() with its k-th allocation failing, k = 0, 1, ..., until it makes
    no more; yields after each failure, which has to be reported as such."""
    for k in range(100):
        lib.fail_after(k)
        try:
            call()
        except art.ArtemisError as e:
            assert e.status == OOM, e
            lib.fail_after(-1)
            yield k
        else:
            assert lib.pending(), "an allocation failed without an error"
            lib.fail_after(-1)
            assert k > 0, "the call allocates nothing"
            return


def _sorted(r, n, seed):
    import torch
    k = np.random.default_rng(seed).integers(0, 2 ** 32, n, dtype=np.uint64).astype(np.uint32)
    kt, vt = torch.from_numpy(k.view(np.int32)).cuda(), torch.arange(n, dtype=torch.int32, device="cuda")
    r.sort_pairs(kt, vt)
    order = np.argsort(k, kind="stable")
    np.testing.assert_array_equal(vt.cpu().numpy(), order)
    np.testing.assert_array_equal(kt.cpu().numpy().view(np.uint32), k[order])


def test_a_reported_failure_is_not_reported_again(art, lib):
    r = art.Renderer()
    lib.fail_after(0)
    with pytest.raises(art.ArtemisError) as e:
        _sorted(r, 5000, 0)
    assert e.value.status == OOM
    _sorted(r, 5000, 0)
    r.close()


def test_sort_scratch(art, lib):
    r = art.Renderer()
    _sorted(r, 5000, 0)
    n = 5000
    for k in _each_failure(art, lib, lambda: _sorted(r, 20000, 1)):
        _sorted(r, n, 2 + k)  # (as many pairs as there was room for before)
        n -= 1000
    _sorted(r, 20000, 9)
    r.close()


def test_sh_coefficients(art, lib):
    """After a load that fails, the plain features are in use."""
    sc = sg.preset("mini")
    oc = sc.octree
    cam = sg.orbit_camera(sc.centroid, 64, 64, az_deg=40.0)
    rng = np.random.default_rng(3)
    coef = [rng.standard_normal((oc.n, (L + 1) ** 2, oc.C)).astype(np.float32) for L in (1, 2)]

    def fresh(L):
        r = renderer(sc)
        set_cam(r, 0, cam)
        set_pose(r, sg.random_pose(2))
        if L:
            r.load_sh_features(L, coef[L - 1])
        return r, render_maps(r, 0, cam, oc.C)

    r, _ = fresh(1)
    plain, want = fresh(0), fresh(2)
    for _ in _each_failure(art, lib, lambda: r.load_sh_features(2, coef[1])):
        for a, b in zip(render_maps(r, 0, cam, oc.C), plain[1]):
            np.testing.assert_array_equal(a, b)
        r.load_sh_features(1, coef[0])
    for a, b in zip(render_maps(r, 0, cam, oc.C), want[1]):
        np.testing.assert_array_equal(a, b)
    for x in (r, plain[0], want[0]):
        x.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
def test_shading_network(art, lib, dtype):
    """After a load that fails there is no network."""
    import torch
    H, W, C = 24, 40, 32
    nets = [sg.unet_weights(k, cin=C) for k in (1, 2)]
    fdt, F_dtype = (torch.float32, "f32") if dtype == "f32" else (torch.bfloat16, "bf16")
    F = torch.from_numpy(np.random.default_rng(1).standard_normal((H, W, C)).astype(np.float32)).cuda().to(fdt)

    def load(r, k):
        r.load_shader(art.ART_NET_UNET, C, sg.UNET_CHANNELS, 4, art.flat_params(nets[k]), dtype)

    def shade(r):
        out = torch.empty((H, W, 4), device="cuda")
        r.shade(0, F, out, F_dtype)
        r.sync_status()
        return out

    def fresh(k):
        r = art.Renderer()
        set_cam(r, 0, sg.orbit_camera((0.0, 0.0, 0.0), W, H))
        load(r, k)
        return r

    r, ref = fresh(0), fresh(1)
    shade(r)
    for _ in _each_failure(art, lib, lambda: load(r, 1)):
        with pytest.raises(art.ArtemisError) as e:
            shade(r)
        assert e.value.status == STATE
    assert torch.equal(shade(r), shade(ref))
    r.close()
    ref.close()


def _posed(art, sc, cams, skip=False):
    r = renderer(sc)
    for v, cam in enumerate(cams):
        set_cam(r, v, cam)
    if skip:
        r.load_proposal((0.05 * np.random.default_rng(5).standard_normal(art.PROPOSAL_PARAMS)).astype(np.float32))
        r.set_config(skip=art.SKIP_LEARNED, max_missed=1e-3, margin=1)
    set_pose(r, sg.random_pose(2))
    return r


@pytest.mark.parametrize("what", ["maps", "skip", "views", "backward", "depth", "labels", "instances"])
def test_buffers_that_grow(art, lib, what):
    """A larger call after a smaller one, with each of its allocations
    failing: the smaller one then gives what it gave, and the larger one, made
    again, what it gives elsewhere."""
    import torch
    sc = sg.preset("mini")
    oc = sc.octree
    cams = [sg.orbit_camera(sc.centroid, W, H, az_deg=40.0) for W, H in ((48, 40), (200, 160))]

    def call(r, k):
        H, W = cams[k].H, cams[k].W
        F, A = torch.empty((H, W, oc.C), device="cuda"), torch.empty((H, W), device="cuda")
        if what == "instances":  # the same view, another capacity of instances
            r.set_config(instance_cap=(1 + k) << 20)
            k = 0
            F, A = F[:cams[0].H, :cams[0].W].contiguous(), A[:cams[0].H, :cams[0].W].contiguous()
        if what in ("maps", "skip", "instances"):
            r.render_feature_maps(k, F, A)
            return [F, A]
        if what == "views":
            G = [torch.empty((c.H, c.W, oc.C), device="cuda") for c in cams]
            r.render_views([0, 1][:k + 1], G[:k + 1])
            return G[:k + 1]
        if what == "depth":
            r.render_depth(k, 0.0, A)
            return [A]
        if what == "labels":
            L = torch.empty((H, W, 3), device="cuda")
            r.render_labels(k, L)
            return [L]
        r.render_feature_maps(k, F, A)
        g = [torch.zeros(t, device="cuda") for t in ((oc.n, oc.C), (oc.n,), (oc.n, 4))]
        r.render_backward(k, F, A, torch.ones_like(F), torch.ones_like(A), *g)
        return g

    def equal(a, b):  # (gradients are summed by atomics)
        return all(torch.allclose(x, y, rtol=1e-4, atol=1e-4 * float(y.abs().max())) if what == "backward"
                   else torch.equal(x, y) for x, y in zip(a, b))

    ref = _posed(art, sc, cams, what == "skip")
    small, large = call(ref, 0), call(ref, 1)
    ref.sync_status()
    for k in range(60):
        r = _posed(art, sc, cams, what == "skip")
        call(r, 0)
        lib.fail_after(k)
        try:
            call(r, 1)
            done = lib.pending()
            assert done, "an allocation failed without an error"
        except art.ArtemisError as e:
            done = False
            assert e.status == OOM, e
        lib.fail_after(-1)
        if not done:
            assert equal(call(r, 0), small), k
        assert equal(call(r, 1), large), k
        r.sync_status()
        r.close()
        if done:
            break
    assert done and k > 0
    ref.close()


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_octree_skeleton_proposal_and_index(art, lib, storage):
    """After a load that fails there is no octree, no skeleton, no pose."""
    import torch
    sc = sg.preset("tiny")
    oc, sk = sc.octree, sc.skeleton
    cam = sg.orbit_camera(sc.centroid, 64, 64, az_deg=40.0)
    F = torch.empty((64, 64, oc.C), device="cuda")

    def octree(r):
        r.load_octree(oc.depth, oc.origin, oc.extent, oc.ijk, oc.joint_idx, oc.weights, oc.features, oc.density, storage)

    def maps(r):
        r.render_feature_maps(0, F)
        return F.clone()

    def refused(f, *a):
        with pytest.raises(art.ArtemisError) as e:
            f(*a)
        assert e.value.status == STATE

    ref = renderer(sc, storage=storage)
    r = renderer(sg.preset("mini"))  # (fewer voxels)
    for x in (ref, r):
        set_cam(x, 0, cam)
        set_pose(x, sg.random_pose(2))
    want = maps(ref)
    maps(r)
    for _ in _each_failure(art, lib, lambda: octree(r)):
        refused(maps, r)
        refused(set_pose, r, sg.random_pose(2))
    for _ in _each_failure(art, lib, lambda: r.load_skeleton(sk.parent, sk.rest)):
        refused(maps, r)
        refused(set_pose, r, sg.random_pose(2))
    set_pose(r, sg.random_pose(2))
    assert torch.equal(maps(r), want)
    for x in (ref, r):
        x.set_config(index=art.INDEX_GRID)
    set_pose(ref, sg.random_pose(2))
    for _ in _each_failure(art, lib, lambda: set_pose(r, sg.random_pose(2))):
        refused(maps, r)
    assert torch.equal(maps(r), maps(ref))
    P = (0.05 * np.random.default_rng(5).standard_normal(art.PROPOSAL_PARAMS)).astype(np.float32)
    bins = [torch.empty((64, 64, 2), dtype=torch.uint8, device="cuda") for _ in range(2)]
    for k in (0, 1, 1):  # (the buffers made before the one that fails stay)
        lib.fail_after(k)
        with pytest.raises(art.ArtemisError) as e:
            r.load_proposal(P)
        assert e.value.status == OOM
        refused(r.run_proposal, 0, bins[0])
    r.load_proposal(P)
    ref.load_proposal(P)
    for x, b in zip((r, ref), bins):
        x.run_proposal(0, b)
        x.sync_status()
    assert torch.equal(*bins)
    ref.close()
    r.close()
