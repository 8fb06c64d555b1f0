"""The radix sort when its look-back waits run out: a build that waits for no
earlier tile (every count not yet published is made from the keys) still
sorts exactly, through both entry points."""
import numpy as np
import pytest

import variants

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def impatient(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return variants.library(tmp_path_factory.mktemp("sort") / "libsort.so", {"binsort.cu": ["-DART_SORT_SPIN=-1"]})


@pytest.mark.parametrize("n", [4097, 8192, 70001, 900001])
@pytest.mark.parametrize("keys", ["equal", "random"])
def test_a_wait_that_runs_out_keeps_the_order(impatient, monkeypatch, n, keys):
    import torch
    import paper_2202_05628_gb300 as art
    monkeypatch.setattr(art, "_lib", impatient)
    rng = np.random.default_rng(n)
    k = rng.integers(0, 2 ** 32, n, dtype=np.uint64).astype(np.uint32) if keys == "random" else np.full(n, 7, np.uint32)
    v = rng.permutation(n).astype(np.uint32)
    order = np.argsort(k, kind="stable")
    r = art.Renderer()
    for sort in (r.sort_pairs, art.sort_pairs_static):
        kt, vt = torch.from_numpy(k.view(np.int32)).cuda(), torch.from_numpy(v.view(np.int32)).cuda()
        assert sort(kt, vt) in (None, 0)
        np.testing.assert_array_equal(kt.cpu().numpy().view(np.uint32), k[order])
        np.testing.assert_array_equal(vt.cpu().numpy().view(np.uint32), v[order])
    r.sync_status()
    r.close()
