"""A batch's host part does not wait for the device: the call returns while the
stream is still busy with what was enqueued before it."""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# instances by value (up to 64 of two strings or more) and from the table, beside
# some of one string
@pytest.mark.parametrize("m", [5, 64, 65, 400])
@pytest.mark.parametrize("graph", [False, True])
def test_batch_call_returns_while_the_stream_is_busy(m, graph):
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(m)
    sizes = r.permutation(np.concatenate([np.ones(20, np.int64), r.choice([2, 40, 600, 3000], m)]))
    first = np.concatenate([[0], np.cumsum(sizes)])
    ss = datagen.from_strings([bytes(x) for x in r.integers(65, 69, (int(first[-1]), 11)).astype(np.uint8)])
    d = sss.to_device(ss)
    n = ss.lens.shape[0]
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    lcp = torch.empty_like(perm)
    prm = sss.params(flags=sss.SSS_FLAG_GRAPH if graph else 0)
    for _ in range(2):  # work memory, staging and graph
        sss.sss_sort_batch(*d, first[:-1], sizes, prm, perm, lcp)
    torch.cuda.synchronize()
    busy = torch.cuda.Event()
    torch.cuda._sleep(200_000_000)  # about 0.1 s
    busy.record()
    sss.sss_sort_batch(*d, first[:-1], sizes, prm, perm, lcp)
    assert not busy.query()
    sss.context().sync()
    perm, lcp = sss.u32(perm), sss.u32(lcp)
    for a, b in list(zip(first[:-1], first[1:]))[::9]:
        sub = datagen.StringSet(ss.chars, ss.offs[a:b], ss.lens[a:b])
        want = oracle.sort(sub)
        assert np.array_equal(perm[a:b], want)
        assert np.array_equal(lcp[a:b], oracle.lcp_array(sub, want))
