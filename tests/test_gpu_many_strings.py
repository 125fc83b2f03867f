"""More strings than a 32-bit number of threads covers with a warp each: the merge of
256 partitions against the sort without partitions."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_150m_strings_in_256_partitions():
    import paper_2404_16517_gb300 as sss
    n = 150_000_000
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    text = torch.empty(n + 12, dtype=torch.uint8, device="cuda").random_(65, 91, generator=g)
    offs = torch.randint(0, n, (n,), generator=g, device="cuda")
    lens = torch.full((n,), 12, dtype=torch.int32, device="cuda")
    ctx = sss.Context()
    perm, lcp, _, _ = sss.sss_sort(text, offs, lens, 256, ctx=ctx)
    want, wl, _, _ = sss.sss_sort(text, offs, lens, 1, ctx=ctx)
    ctx.sync()
    assert torch.equal(perm, want)
    assert torch.equal(lcp, wl)
    ctx.close()
    del text, offs, lens, perm, lcp, want, wl
    torch.cuda.empty_cache()
