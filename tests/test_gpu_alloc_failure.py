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
