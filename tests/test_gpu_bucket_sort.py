"""The in-CTA sort by buckets and ranks: key distributions that spread and that do
not (merge sort), at the edges of its CTA sizes, against the oracle."""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _strings(kind, n, r):
    if kind == "uniform":      # dense characters, one head
        return [bytes(r.integers(65, 91, 12).astype(np.uint8)) for _ in range(n)]
    if kind == "bytes":        # all byte values but 0, every length
        return [bytes(r.integers(1, 256, r.integers(0, 9)).astype(np.uint8)) for _ in range(n)]
    if kind == "skewed":       # clusters: 90% of the characters are one value
        return [bytes(np.where(r.random(14) < 0.9, 80, r.integers(65, 91, 14)).astype(np.uint8)) for _ in range(n)]
    if kind == "equal":        # few distinct strings
        return [b"AB" * 10 + bytes([65 + int(r.integers(0, 3))]) for _ in range(n)]
    if kind == "staircase":    # many heads: every string leaves one template elsewhere
        t = bytes(r.integers(65, 69, 400).astype(np.uint8))
        out = []
        for _ in range(n):
            c = int(r.integers(0, 400))
            out.append(t[:c] + bytes(r.integers(65, 69, int(r.integers(0, 10))).astype(np.uint8)))
        return out
    if kind == "ended":        # strings that end where others go on
        t = b"Q" * 300
        return [t[:int(r.integers(290, 301))] + (b"" if r.random() < 0.5 else bytes([int(r.integers(64, 67))]))
                for _ in range(n)]
    raise ValueError(kind)


@pytest.mark.parametrize("kind", ["uniform", "bytes", "skewed", "equal", "staircase", "ended"])
# whole segments of the bucket CTA (to 4,352) and of the large one (to 8,192), with
# the merge sort's capacity (4,096) between, and a partitioned one
@pytest.mark.parametrize("n", [2049, 4095, 4097, 4352, 4353, 8192, 8193])
def test_sizes_and_distributions(kind, n):
    import paper_2404_16517_gb300 as sss
    ss = datagen.from_strings(_strings(kind, n, np.random.default_rng(n)))
    chars, offs, lens = sss.to_device(ss)
    want = oracle.sort(ss)
    wl = oracle.lcp_array(ss, want)
    for prm in (sss.params(), sss.params(bucket_target=256, cta_cap=64)):
        perm, lcp, _, _ = sss.sss_sort(chars, offs, lens, prm=prm)
        sss.context().sync()
        assert np.array_equal(sss.u32(perm), want)
        assert np.array_equal(sss.u32(lcp), wl)


# the CTA finisher's first iteration (65 .. 2,048 strings), as the only segment of a
# call (its 128- and 512-thread instances) and as partitions beside others
@pytest.mark.parametrize("kind", ["uniform", "bytes", "skewed", "equal", "staircase", "ended"])
@pytest.mark.parametrize("n", [65, 127, 511, 512, 513, 1000, 2047, 2048])
def test_finisher_sizes_and_distributions(kind, n):
    import paper_2404_16517_gb300 as sss
    ss = datagen.from_strings(_strings(kind, n, np.random.default_rng(n + 1)))
    chars, offs, lens = sss.to_device(ss)
    for p in (1, 3):
        rp, rl = sss.sss_local_sort(chars, offs, lens, p)
        sss.context().sync()
        want, wl = oracle.local_sort(ss, p)
        assert np.array_equal(sss.u32(rp), want)
        assert np.array_equal(sss.u32(rl), wl)
