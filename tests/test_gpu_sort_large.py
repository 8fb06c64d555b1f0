"""The radix sort at the size from which its look-back words hold 64 bits."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(1 << 28) - 1, (1 << 28) + 4099])
def test_sorts_stably(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2202_05628_gb300 as art
    g = torch.Generator(device="cuda").manual_seed(n)
    # (some keys many times, so that the order of equal ones shows)
    k = torch.randint(0, 1 << 26, (n,), device="cuda", generator=g, dtype=torch.int32) * 31
    ks, vs = k.clone(), torch.arange(n, device="cuda", dtype=torch.int32)
    r = art.Renderer()
    r.sort_pairs(ks, vs, 32)
    r.sync_status()
    r.close()
    assert torch.equal(ks, k[vs.long()])
    d = ks.long() & 0xFFFFFFFF
    up = d[1:] > d[:-1]
    same = d[1:] == d[:-1]
    assert bool((up | (same & (vs[1:] > vs[:-1]))).all())
    assert bool(same.any())
