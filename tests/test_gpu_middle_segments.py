"""Segments between a bucket CTA's capacity and the largest one sorted whole: sorted
whole, or partitioned when there are few of them (more are few beside larger ones);
both ways, on both sides of the lines and at the sizes' edges, against the oracle."""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _line(larger):
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    return 2 * sm if larger else sm // 8


# (larger segments, strings of a middle one, middle ones relative to the line or as such)
@pytest.mark.parametrize("larger,size,k", [(0, 4353, 1), (0, 8192, 3), (0, 4400, "line"), (0, 4400, "line+1"),
                                           (1, 4352, 2), (1, 4353, 1), (1, 8192, 2),
                                           (1, 4400, "line"), (1, 4400, "line+1"), (3, 5003, 40)])
@pytest.mark.parametrize("target", [0, 1024])
def test_middle_segments(larger, size, k, target):
    import paper_2404_16517_gb300 as sss
    if isinstance(k, str):
        k = _line(larger) + (1 if k == "line+1" else 0)
    r = np.random.default_rng([larger, size, k])
    sizes = r.permutation(np.array([8193, 20011, 30000][:larger] + [size] * k + [3, 300, 2500]))
    first = np.concatenate([[0], np.cumsum(sizes)])
    n = int(first[-1])
    lens = r.integers(3, 12, n).astype(np.uint32)
    offs = (np.arange(n) * 12).astype(np.uint64)
    chars = r.integers(65, 70, 12 * n).astype(np.uint8)
    chars.reshape(n, 12)[r.random(n) < 0.3, :3] = 66
    ss = datagen.StringSet(chars, offs, lens)
    d = sss.to_device(ss)
    ref = None
    for knobs in ({}, {"direct_cap": 8192}, {"direct_cap": 4352}):
        perm, lcp, _ = sss.sss_sort_batch(*d, first[:-1], sizes, sss.params(bucket_target=target, **knobs))
        sss.context().sync()
        got = sss.u32(perm), sss.u32(lcp)
        if ref is None:
            ref = got
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), knobs
    for a, b in list(zip(first[:-1], first[1:]))[::1 + len(sizes) // 12]:
        sub = datagen.StringSet(ss.chars, ss.offs[a:b], ss.lens[a:b])
        want = oracle.sort(sub)
        assert np.array_equal(ref[0][a:b], want)
        assert np.array_equal(ref[1][a:b], oracle.lcp_array(sub, want))
