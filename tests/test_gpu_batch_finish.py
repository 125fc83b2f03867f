"""The last pass of a batch (instance-local indices, dist) around its span of 2,048
positions a CTA, with instances that start at odd positions."""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[1, 255, 256, 257, 2047, 2048, 2049, 4097], [5000], [3] * 700, [2049] * 3 + [1]])
def test_spans(sizes):
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(len(sizes))
    n = sum(sizes)
    ss = datagen.from_strings([bytes(r.integers(65, 69, int(r.integers(1, 9))).astype(np.uint8)) for _ in range(n)])
    chars, offs, lens = sss.to_device(ss)
    first = np.concatenate([[0], np.cumsum(sizes)])
    perm, lcp, dist = sss.sss_sort_batch(chars, offs, lens, first[:-1], np.array(sizes), want_dist=True)
    sss.context().sync()
    P, L, D = sss.u32(perm), sss.u32(lcp), sss.u32(dist)
    for a, b in zip(first[:-1], first[1:]):
        sub = datagen.StringSet(ss.chars, ss.offs[a:b], ss.lens[a:b])
        want = oracle.sort(sub)
        wl = oracle.lcp_array(sub, want)
        assert np.array_equal(P[a:b], want)
        assert np.array_equal(L[a:b], wl)
        assert np.array_equal(D[a:b], oracle.dist(sub, want, wl))
