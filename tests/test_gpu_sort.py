"""The radix sort's edges: tiles of 4096 pairs (one short, exact, one over,
several look-back rounds of 16 tiles), keys that share digits, every width."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n", [2, 33, 4096, 8191, 70001, 900001])
@pytest.mark.parametrize("keys,bits", [("equal", 32), ("two", 32), ("tiles", 32), ("random", 24), ("random", 8)])
def test_sorts_stably(n, keys, bits):
    import torch
    import paper_2202_05628_gb300 as art
    rng = np.random.default_rng(n)
    k = {"equal": lambda: np.full(n, 0xDEADBEEF, np.uint32),
         "two": lambda: rng.integers(0, 2, n).astype(np.uint32) * np.uint32(0xFF00FF01),
         "tiles": lambda: ((rng.integers(0, 300, n) // 7 * 7 << 17) | rng.integers(0, 1 << 17, n)).astype(np.uint32),
         "random": lambda: rng.integers(0, 2 ** 32, n, dtype=np.uint64).astype(np.uint32)}[keys]()
    v = rng.permutation(n).astype(np.uint32)
    order = np.argsort(k.astype(np.uint64) & np.uint64((1 << bits) - 1), kind="stable")
    r = art.Renderer()
    for sort in (lambda a, b: r.sort_pairs(a, b, bits), lambda a, b: art.sort_pairs_static(a, b, bits)):
        kt, vt = torch.from_numpy(k.view(np.int32)).cuda(), torch.from_numpy(v.view(np.int32)).cuda()
        for _ in range(2):  # the second call finds the first one's scratch
            kt.copy_(torch.from_numpy(k.view(np.int32)))
            vt.copy_(torch.from_numpy(v.view(np.int32)))
            assert sort(kt, vt) in (None, 0)
        np.testing.assert_array_equal(kt.cpu().numpy().view(np.uint32), k[order])
        np.testing.assert_array_equal(vt.cpu().numpy().view(np.uint32), v[order])
    r.sync_status()
