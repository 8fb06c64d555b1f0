"""A grown buffer that gets its old address back is as new: what has to start
at zero does.  The library is linked with a cudaMalloc that rounds up, and
returns the block freed last, filled with 2s, where that is large enough."""
import numpy as np
import pytest

import scenegen as sg
import variants
from helpers import render_maps, renderer, set_cam, set_pose

pytestmark = pytest.mark.gpu

REUSING_MALLOC = """
#include <stddef.h>
#include <stdint.h>
int __real_cudaMalloc(void** p, size_t n);
int __real_cudaFree(void* p);
int cudaMemcpy(void* dst, const void* src, size_t n, int kind);
enum { kBlock = 1 << 23, kMany = 4096 };
static void* own[kMany];
static int owned;
static void* freed;
int __wrap_cudaFree(void* p) {
  for (int i = 0; p && i < owned; ++i)
    if (own[i] == p && !freed) {
      freed = p;
      return 0;
    }
  return __real_cudaFree(p);
}
int __wrap_cudaMalloc(void** p, size_t n) {
  static uint32_t twos[kBlock / 4];
  if (n > kBlock || owned == kMany) return __real_cudaMalloc(p, n);
  if (freed) {
    *p = freed;
    freed = 0;
    for (int i = 0; i < kBlock / 4; ++i) twos[i] = 2;
    return cudaMemcpy(*p, twos, kBlock, 1);
  }
  const int e = __real_cudaMalloc(p, kBlock);
  if (!e) own[owned++] = *p;
  return e;
}
"""


def test_exact_rewalk_flags_start_over(tmp_path, monkeypatch):
    """The second render's stamp is 2: tiles flagged with it by chance would
    not be queued for the exact walk."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2202_05628_gb300 as art
    rng = np.random.default_rng(17)
    n = 40  # coincident voxels: more hits at one distance than a pixel's reorder buffer holds
    w = np.zeros((n, 4), np.float32)
    w[:, 0] = 1.0
    oc = sg.Octree(4, np.array([-0.5, -0.5, -0.5], np.float32), 1.0, np.full((n, 3), 8, np.uint16),
                   np.zeros((n, 4), np.uint8), w, rng.standard_normal((n, 8)).astype(np.float32),
                   rng.uniform(1.0, 3.0, n).astype(np.float32), np.zeros(n, np.float32))
    sc = sg.Scene(oc, sg.Skeleton(np.array([-1], np.int32), np.zeros((1, 3), np.float32)), np.zeros(3), 1.0, None, None)
    c = oc.centers()[0].astype(np.float64)
    M = sg.look_at(c + np.array([0.07, 0.11, -1.0]), c)
    small, large = (sg.Camera(W, 16, 120.0, 120.0, W / 2, 8.0, M, 0.1, 3.0) for W in (24, 240))

    def frames(lib, cams):
        with monkeypatch.context() as m:
            if lib:
                m.setattr(art, "_lib", lib)
            r = renderer(sc)
            set_pose(r, sg.rest_pose(1))
            for cam in cams:
                set_cam(r, 0, cam)
                F, _ = render_maps(r, 0, cam, 8)
            st = r.sync_status()
            r.close()
        return F, st["exact_tiles"]

    want = frames(None, [large])
    got = frames(variants.library(tmp_path / "libreuse.so", wrap=["cudaMalloc", "cudaFree"], source=REUSING_MALLOC),
                 [small, large])
    assert want[1] > 0 and got[1] == want[1]
    np.testing.assert_array_equal(got[0], want[0])
