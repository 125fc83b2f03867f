"""One context on several streams: its calls share work memory and device state and
run one after the other whatever their streams."""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _set(n, seed):
    """n strings, a part of them equal, a part with a long shared prefix."""
    r = np.random.default_rng(seed)
    lens = (r.integers(0, 13, n) + np.where(r.random(n) < 0.2, 40, 0)).astype(np.uint32)
    offs = np.zeros(n, np.uint64)
    offs[1:] = np.cumsum(lens[:-1].astype(np.uint64))
    chars = r.integers(65, 69, int(lens.astype(np.int64).sum()) + 1).astype(np.uint8)
    long = lens >= 40
    chars[offs[long].astype(np.int64)[:, None] + np.arange(38)[None, :]] = 66
    return datagen.StringSet(chars, offs, lens)


# sizes of a CTA, of one grid class and of two, with and without partitions
@pytest.mark.parametrize("sizes", [[(30011, 1), (70001, 1)], [(300007, 1), (5000, 1)], [(200003, 1), (150001, 4)],
                                   [(40009, 3), (90001, 16)], [(1500, 1), (60001, 1)]])
def test_default_context_on_two_streams(sizes):
    import paper_2404_16517_gb300 as sss
    sets = [_set(n, n) for n, _ in sizes]
    dev = [sss.to_device(s) for s in sets]
    streams = [torch.cuda.Stream() for _ in sets]
    torch.cuda.synchronize()
    out = []
    for _ in range(4):
        for st, d, (n, p) in zip(streams, dev, sizes):
            with torch.cuda.stream(st):
                out.append(sss.sss_sort(*d, p)[:2])
    torch.cuda.synchronize()
    sss.context().sync()
    want = [oracle.sort(s) for s in sets]
    lcp = [oracle.lcp_array(s, w) for s, w in zip(sets, want)]
    for i, (perm, l) in enumerate(out):
        assert np.array_equal(sss.u32(perm), want[i % 2]), i
        assert np.array_equal(sss.u32(l), lcp[i % 2]), i


def test_batches_and_suffixes_on_two_streams():
    import paper_2404_16517_gb300 as sss
    sizes = [3000, 70, 9000, 2, 2500] * 20
    first = np.concatenate([[0], np.cumsum(sizes)])
    ss = _set(int(first[-1]), 11)
    d = sss.to_device(ss)
    text = np.tile(np.random.default_rng(1).integers(65, 70, 300).astype(np.uint8), 90)
    t = torch.from_numpy(text).cuda()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    out = []
    for _ in range(3):
        with torch.cuda.stream(a):
            x = sss.sss_sort_batch(*d, first[:-1], sizes)[:2]
        with torch.cuda.stream(b):
            out.append((x, sss.sss_suffix_sort(t)))
    torch.cuda.synchronize()
    n = text.shape[0]
    sfx = datagen.StringSet(text, np.arange(n, dtype=np.uint64), np.arange(n, 0, -1).astype(np.uint32))
    want = oracle.sort(sfx)
    wl = oracle.lcp_array(sfx, want)
    for (perm, lcp), (sa, sl) in out:
        assert np.array_equal(sss.u32(sa), want) and np.array_equal(sss.u32(sl), wl)
        perm, lcp = sss.u32(perm), sss.u32(lcp)
        for lo, hi in list(zip(first[:-1], first[1:]))[::7]:
            sub = datagen.StringSet(ss.chars, ss.offs[lo:hi], ss.lens[lo:hi])
            w = oracle.sort(sub)
            assert np.array_equal(perm[lo:hi], w) and np.array_equal(lcp[lo:hi], oracle.lcp_array(sub, w))


def test_the_second_stream_waits_on_the_device():
    """The host goes on at once, the second call's work follows the first's."""
    import paper_2404_16517_gb300 as sss
    sets = [_set(60001, 1), _set(60001, 2)]
    dev = [sss.to_device(s) for s in sets]
    streams = [torch.cuda.Stream() for _ in sets]
    ends = [torch.cuda.Event() for _ in sets]
    for d in dev:
        sss.sss_sort(*d)
    torch.cuda.synchronize()
    out = []
    for i in range(2):
        with torch.cuda.stream(streams[i]):
            if i == 0:
                torch.cuda._sleep(200_000_000)  # about 0.1 s
            out.append(sss.sss_sort(*dev[i])[:2])
            ends[i].record()
    assert not ends[0].query()
    ends[1].synchronize()
    assert ends[0].query()
    for s, (perm, lcp) in zip(sets, out):
        want = oracle.sort(s)
        assert np.array_equal(sss.u32(perm), want) and np.array_equal(sss.u32(lcp), oracle.lcp_array(s, want))


# one CTA's sort, and a few lists by their classes: the calls that need no rounds
@pytest.mark.parametrize("p", [1, 3])
def test_calls_without_rounds_can_be_captured(p):
    """On the capturing stream a call neither waits for the context's earlier calls
    nor marks its end; the graph sorts what the buffers hold when it is launched."""
    import paper_2404_16517_gb300 as sss
    sets = [_set(1500, s) for s in (21, 22)]
    cap = max(s.chars.shape[0] for s in sets)
    dev = [sss.to_device(s) for s in sets]
    chars = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    offs, lens = torch.empty_like(dev[0][1]), torch.empty_like(dev[0][2])
    perm = torch.empty(1500, dtype=torch.int32, device="cuda")
    lcp = torch.empty_like(perm)

    def load(d):
        chars[:d[0].numel()].copy_(d[0])
        offs.copy_(d[1])
        lens.copy_(d[2])

    load(dev[0])
    sss.sss_local_sort(chars, offs, lens, p, None, perm, lcp)  # work memory and kernels
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sss.sss_local_sort(chars, offs, lens, p, None, perm, lcp)
    for s, d in zip(sets, dev):
        load(d)
        graph.replay()
        torch.cuda.synchronize()
        sss.context().sync()
        want, wl = oracle.local_sort(s, p)
        assert np.array_equal(sss.u32(perm), want)
        assert np.array_equal(sss.u32(lcp), wl)
        sss.sss_sort(*d, 2)  # and calls outside the graph go on
        sss.context().sync()
