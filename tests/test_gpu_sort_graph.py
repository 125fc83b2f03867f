"""The local sort as one graph launch: its kernels read the call's pointers and
sizes from device memory, so one graph serves calls of any inputs and work
memory; grids, tile lookup and the initial segments' way to the device depend
on the sizes."""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _set(n, seed):
    """n short strings over a small alphabet (many equal), a fifth of them with a
    long shared prefix."""
    r = np.random.default_rng(seed)
    lens = r.integers(0, 13, n)
    long = r.random(n) < 0.2
    lens = np.where(long, lens + 40, lens).astype(np.uint32)
    offs = np.zeros(n, np.uint64)
    offs[1:] = np.cumsum(lens[:-1].astype(np.uint64))
    chars = r.integers(65, 69, int(lens.astype(np.int64).sum()) + 1).astype(np.uint8)
    pos = offs[long].astype(np.int64)[:, None] + np.arange(38)[None, :]
    chars[pos] = 66
    return datagen.StringSet(chars, offs, lens)


def _check(ss, perm, lcp, a=0, b=None):
    sub = datagen.StringSet(ss.chars, ss.offs[a:b], ss.lens[a:b])
    want = oracle.sort(sub)
    assert np.array_equal(perm[a:b], want)
    assert np.array_equal(lcp[a:b], oracle.lcp_array(sub, want))


# below and above the sizes where the grids change, the last with listed tiles
@pytest.mark.parametrize("n", [2049, (1 << 17), (1 << 17) + 1, (1 << 18) + 1, (1 << 19) + 1])
def test_grid_classes(n):
    import paper_2404_16517_gb300 as sss
    ss = _set(n, n)
    chars, offs, lens = sss.to_device(ss)
    perm, lcp, _, _ = sss.sss_sort(chars, offs, lens)
    sss.context().sync()
    _check(ss, sss.u32(perm), sss.u32(lcp))


# initial segments by value (<= 64) and through the device table, of every class
@pytest.mark.parametrize("m", [1, 64, 65, 300])
def test_initial_segments(m):
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(m)
    sizes = r.choice([1, 2, 4, 5, 32, 33, 64, 65, 512, 513, 2048, 2049, 9000], m)
    first = np.concatenate([[0], np.cumsum(sizes)])
    ss = _set(int(first[-1]) + 1, 7 + m)
    chars, offs, lens = sss.to_device(ss)
    for _ in range(2):
        perm, lcp, _ = sss.sss_sort_batch(chars, offs, lens, first[:-1], sizes)
        sss.context().sync()
        p, l = sss.u32(perm), sss.u32(lcp)
        for k in range(0, m, 1 + m // 40):
            _check(ss, p, l, int(first[k]), int(first[k + 1]))


def test_one_by_one_launches_give_the_same():
    """With kernel timing on the same kernels are launched one by one."""
    import paper_2404_16517_gb300 as sss
    ss = _set(60001, 3)
    chars, offs, lens = sss.to_device(ss)
    ctx = sss.Context()
    ref = [t.clone() for t in sss.sss_sort(chars, offs, lens, 5, ctx=ctx)[:2]]
    ctx.set_timing(True)
    got = sss.sss_sort(chars, offs, lens, 5, ctx=ctx)[:2]
    ctx.sync()
    assert all(torch.equal(a, b) for a, b in zip(ref, got))
    assert "ls_lg_plan" in ctx.kernel_stats()
    ctx.close()


def test_contexts_side_by_side():
    """Two contexts on two streams, each with its own device state."""
    import paper_2404_16517_gb300 as sss
    sets = [_set(30011, 1), _set(70001, 2)]
    dev = [sss.to_device(s) for s in sets]
    streams = [torch.cuda.Stream() for _ in sets]
    torch.cuda.synchronize()
    ctx, out = [], []
    for st in streams:
        with torch.cuda.stream(st):
            ctx.append(sss.Context())
    for _ in range(3):
        out = []
        for st, c, d in zip(streams, ctx, dev):
            with torch.cuda.stream(st):
                out.append(sss.sss_sort(*d, 3, ctx=c))
    for c, s, o in zip(ctx, sets, out):
        c.sync()
        _check(s, sss.u32(o[0]), sss.u32(o[1]))
        c.close()


# periods that leave groups of equal ranks in every size class (pairs to > 2,048)
@pytest.mark.parametrize("period,copies,max_len", [(700, 2, 0), (250, 30, 0), (100, 70, 1000), (20, 700, 0), (3, 2900, 0),
                                                   (7, 1300, 129)])
def test_suffix_groups_of_every_class(period, copies, max_len):
    """The rank doubling of the suffix sort refines groups in place."""
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(period)
    text = np.tile(r.integers(65, 70, period).astype(np.uint8), copies)
    text[-5:] = 80
    n = text.shape[0]
    lens = np.arange(n, 0, -1).astype(np.uint32)
    ss = datagen.StringSet(text, np.arange(n, dtype=np.uint64), np.minimum(lens, max_len or n).astype(np.uint32))
    sa, lcp = sss.sss_suffix_sort(torch.from_numpy(text).cuda(), max_len)
    sss.context().sync()
    _check(ss, sss.u32(sa), sss.u32(lcp))


# shared prefixes around the cached reference characters, units of a quarter and
# of a whole tile
@pytest.mark.parametrize("n", [3000, 40000])
@pytest.mark.parametrize("shared", [500, 1015, 1024, 1031, 2100])
def test_keys_past_the_cached_reference(n, shared):
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(n + shared)
    lens = (shared - 9 + r.integers(0, 30, n)).astype(np.uint32)
    offs = np.zeros(n, np.uint64)
    offs[1:] = np.cumsum(lens[:-1].astype(np.uint64))
    chars = r.integers(65, 69, int(lens.astype(np.int64).sum()) + 1).astype(np.uint8)
    t = r.integers(65, 91, shared).astype(np.uint8)
    chars[offs.astype(np.int64)[:, None] + np.arange(shared - 12)[None, :]] = t[:shared - 12]
    ss = datagen.StringSet(chars, offs, lens)
    d = sss.to_device(ss)
    perm, lcp, _, _ = sss.sss_sort(*d)
    sss.context().sync()
    _check(ss, sss.u32(perm), sss.u32(lcp))


# buckets of equal keys around the size that is copied by all CTAs (2^17): equal
# strings, and strings that go on past an equal key
@pytest.mark.parametrize("m", [(1 << 17) - 3, (1 << 17) + 2, 300007])
@pytest.mark.parametrize("kind", ["ended", "goes on"])
def test_largest_equality_buckets(m, kind):
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(m)
    if kind == "ended":
        strs = [b"EQUAL"] * m + [bytes(x) for x in r.integers(65, 91, (5000, 7)).astype(np.uint8)]
    else:  # whichever half the reference is from, the other one's keys are equal
        t = r.integers(65, 91, (2 * m, 3)).astype(np.uint8)
        strs = [(b"B" if i & 1 else b"C") * 20 + t[i].tobytes() for i in range(2 * m)]
    ss = datagen.from_strings([strs[i] for i in r.permutation(len(strs))])
    chars, offs, lens = sss.to_device(ss)
    perm, lcp, _, _ = sss.sss_sort(chars, offs, lens)
    sss.context().sync()
    _check(ss, sss.u32(perm), sss.u32(lcp))
