"""Sub-splitter bounds of the merge: windows on both sides of a lane per string
(p small and large), strings that share more with a sub-splitter than a lane
compares, many equal strings, pieces with few samples or none."""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _set(kind, n, r):
    tail = r.integers(65, 91, (n, 6)).astype(np.uint8)
    if kind == "templates":  # shared prefixes of up to 300 characters, three of them
        t = r.integers(65, 91, (3, 300)).astype(np.uint8)
        pick, cut = r.integers(0, 3, n), r.integers(250, 301, n)
        return [t[p, :c].tobytes() + x.tobytes() for p, c, x in zip(pick, cut, tail)]
    if kind == "equal":      # long equal strings, a few hundred distinct ones
        base = [b"L" * 90 + bytes(r.integers(65, 68, 5).astype(np.uint8)) for _ in range(300)]
        return [base[i] for i in r.integers(0, 300, n)]
    return [x.tobytes()[:int(l)] for x, l in zip(tail, r.integers(1, 7, n))]  # short ones


@pytest.mark.parametrize("kind", ["templates", "equal", "short"])
@pytest.mark.parametrize("n,p", [(9001, 2), (20011, 4), (40009, 16), (30011, 64), (3001, 100)])
def test_merge_windows(kind, n, p):
    import paper_2404_16517_gb300 as sss
    ss = datagen.from_strings(_set(kind, n, np.random.default_rng(n + p)))
    chars, offs, lens = sss.to_device(ss)
    perm, lcp, _, _ = sss.sss_sort(chars, offs, lens, p)
    sss.context().sync()
    want = oracle.sort(ss)
    assert np.array_equal(sss.u32(perm), want)
    assert np.array_equal(sss.u32(lcp), oracle.lcp_array(ss, want))


# stage C alone: samples ranked in pairs (to 256) and sorted (above), runs around the
# 33-way split, with and without truncation
@pytest.mark.parametrize("kind", ["templates", "equal", "short"])
@pytest.mark.parametrize("n,p,v", [(5, 8, 2), (64, 2, 1), (33 * 4, 4, 2), (34 * 4 + 1, 4, 3), (20011, 16, 15),
                                   (20011, 16, 16), (9001, 64, 3), (70001, 3, 2)])
def test_partition(kind, n, p, v):
    import paper_2404_16517_gb300 as sss
    ss = datagen.from_strings(_set(kind, n, np.random.default_rng(n + p + v)))
    rp, _ = oracle.local_sort(ss, p)
    chars, offs, lens = sss.to_device(ss)
    t_rp = torch.from_numpy(rp.view(np.int32)).cuda()
    for tr in (None, oracle.doubling(ss, 0, oracle.default_kmax(ss), 0)):
        _, want_spl = oracle.splitters(ss, oracle.samples(rp, n, p, v), p, tr)
        want_b = oracle.bounds(ss, rp, p, want_spl, tr)
        t_tr = None if tr is None else torch.from_numpy(tr.view(np.int32)).cuda()
        spl, bnd = sss.sss_partition(chars, offs, lens, t_rp, p, trunc=t_tr, prm=sss.params(v=v))
        sss.context().sync()
        assert np.array_equal(sss.u32(spl), want_spl)
        assert np.array_equal(sss.u32(bnd).reshape(-1), want_b.reshape(-1))


# a few distinct strings only: runs of equal samples longer than a warp, slices of
# one to hundreds of chunks of 32 records
@pytest.mark.parametrize("n,p", [(33, 2), (5000, 2), (70001, 4), (70001, 16)])
@pytest.mark.parametrize("distinct", [1, 3])
def test_long_equal_runs(n, p, distinct):
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(n + p)
    base = [b"M" * 30 + bytes([65 + i]) for i in range(distinct)]
    ss = datagen.from_strings([base[i] for i in r.integers(0, distinct, n)])
    chars, offs, lens = sss.to_device(ss)
    perm, lcp, _, _ = sss.sss_sort(chars, offs, lens, p)
    sss.context().sync()
    want = oracle.sort(ss)
    assert np.array_equal(sss.u32(perm), want)
    assert np.array_equal(sss.u32(lcp), oracle.lcp_array(ss, want))
