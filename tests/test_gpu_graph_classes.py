"""The sort's graph, its kernels launched one by one, and the oracle agree: in every
grid class, with both bucket CTAs, with partitions and as a batch."""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _set(n, seed):
    """n strings over four letters, 0 to 12 characters after a prefix that about half
    of them share."""
    r = np.random.default_rng(seed)
    own = r.integers(0, 13, n)
    shared = np.where(r.random(n) < 0.5, 30, 0)
    lens = (own + shared).astype(np.uint32)
    offs = np.zeros(n, np.uint64)
    offs[1:] = np.cumsum(lens[:-1].astype(np.uint64))
    chars = r.integers(65, 69, int(lens.astype(np.int64).sum()) + 1).astype(np.uint8)
    chars[offs[shared > 0].astype(np.int64)[:, None] + np.arange(30)[None, :]] = 67
    return datagen.StringSet(chars, offs, lens)


def _runs(sss, call):
    """The call's (perm, lcp) as one graph launch, with timing off and on, and as
    single launches; and whether each was what it should be."""
    out = []
    for timing, flags, name in ((False, 0, "ls_graph"), (True, sss.SSS_FLAG_GRAPH, "ls_graph"), (True, 0, "ls_lg_plan")):
        ctx = sss.Context()
        ctx.set_timing(timing)
        for _ in range(2):  # a first call and one of the kept graph
            perm, lcp = call(ctx, flags)
        ctx.sync()
        stats = ctx.kernel_stats()
        assert name in stats and ("ls_graph" in stats) == (name == "ls_graph")
        out.append((sss.u32(perm), sss.u32(lcp)))
        ctx.close()
    return out


# the sizes end the grid classes; bucket_target 1024 takes the 256-thread bucket CTA
@pytest.mark.parametrize("n", [60001, 1 << 17, (1 << 17) + 1, 1 << 18, (1 << 18) + 1, 1 << 19, (1 << 19) + 1])
@pytest.mark.parametrize("target", [1024, 2048])
def test_sort(n, target):
    import paper_2404_16517_gb300 as sss
    ss = _set(n, n)
    d = sss.to_device(ss)
    want = oracle.sort(ss)
    wl = oracle.lcp_array(ss, want)
    for p in (1, 3):
        for perm, lcp in _runs(sss, lambda ctx, flags: sss.sss_sort(
                *d, p, sss.params(flags=flags, bucket_target=target), ctx=ctx)[:2]):
            assert np.array_equal(perm, want)
            assert np.array_equal(lcp, wl)


@pytest.mark.parametrize("scale", [1, 3, 6, 12])
@pytest.mark.parametrize("target", [1024, 2048])
def test_batch(scale, target):
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(scale)
    sizes = r.permutation(np.array([2, 5, 40, 300, 700, 2049, 4353, 9000, 30000] * scale + [60000]))
    first = np.concatenate([[0], np.cumsum(sizes)])
    ss = _set(int(first[-1]), scale)
    d = sss.to_device(ss)
    runs = _runs(sss, lambda ctx, flags: sss.sss_sort_batch(
        *d, first[:-1], sizes, sss.params(flags=flags, bucket_target=target), ctx=ctx)[:2])
    for a, b in zip(first[:-1], first[1:]):
        sub = datagen.StringSet(ss.chars, ss.offs[a:b], ss.lens[a:b])
        want = oracle.sort(sub)
        wl = oracle.lcp_array(sub, want)
        for perm, lcp in runs:
            assert np.array_equal(perm[a:b], want)
            assert np.array_equal(lcp[a:b], wl)
