"""Strings that are extensions of others, above all of a segment's reference when
that one has 2^k - 1 characters left: its key and an extension's then share their
head, and only the extension has characters.  Against the oracle, through the
finishers, the whole-segment and the partitioned sorts, with partitions and as a
batch."""
import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _same_length(n, length, digits, base, one_in, r):
    """n strings of `length` characters, a shared prefix and then digits of the
    given base; one in `one_in` is another one followed by the smallest digit, at
    a lower or a higher index.  No string is a shorter prefix of another."""
    t = bytes(r.integers(65, 91, length - digits).astype(np.uint8))
    d = (48 + r.integers(0, base, (n, digits))).astype(np.uint8)
    out = [t + x.tobytes() for x in d]
    for i in r.choice(n, max(1, n // one_in), replace=False):
        out[int(i)] = out[int(r.integers(n))][:length] + b"0"
    return out


def _check(strs, p_list, prms):
    import paper_2404_16517_gb300 as sss
    ss = datagen.from_strings(strs)
    chars, offs, lens = sss.to_device(ss)
    want = oracle.sort(ss)
    wl = oracle.lcp_array(ss, want)
    for p in p_list:
        for prm in prms:
            perm, lcp, _, _ = sss.sss_sort(chars, offs, lens, p, prm)
            sss.context().sync()
            assert np.array_equal(sss.u32(perm), want), (p, prm.bucket_target)
            assert np.array_equal(sss.u32(lcp), wl), (p, prm.bucket_target)


def _prms(sss):
    return [sss.params(), sss.params(bucket_target=1024, cta_cap=64, direct_cap=8192)]


# finishers (65 .. 2,048 strings), bucket CTAs (to 4,352), whole segments (to 8,192)
# and partitions; the strings are about as many as the values of their digits, so
# that some of them is an extension of whichever is the reference
@pytest.mark.parametrize("n", [65, 500, 512, 513, 2048, 2049, 4352, 4353, 8192, 8193, 20000])
@pytest.mark.parametrize("length", [7, 15, 63, 255])
def test_reference_of_a_power_of_two_less_one(n, length):
    import paper_2404_16517_gb300 as sss
    base = 2 if length > 7 else max(2, int(round((0.5 * n) ** (1 / 7))))
    digits = 7 if length == 7 else min(length, max(4, n.bit_length() - 2))
    for seed in range(6):
        r = np.random.default_rng([n, length, seed])
        _check(_same_length(n, length, digits, base, 12, r), (1,), _prms(sss))


@pytest.mark.parametrize("n", [2000, 20000])
@pytest.mark.parametrize("length", [7, 15, 255])
def test_extensions_in_partitions(n, length):
    import paper_2404_16517_gb300 as sss
    base = 2 if length > 7 else max(2, int(round((0.5 * n) ** (1 / 7))))
    digits = 7 if length == 7 else n.bit_length() - 3
    for seed in range(6):
        r = np.random.default_rng([n, length, seed, 1])
        _check(_same_length(n, length, digits, base, 12, r), (4,), _prms(sss))


def test_extensions_in_a_batch():
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(5)
    sizes = r.choice([70, 300, 500, 600, 2000, 3000, 9000], 90)
    first = np.concatenate([[0], np.cumsum(sizes)])
    strs = []
    for s in sizes:
        strs += _same_length(int(s), 15, max(4, int(s).bit_length() - 2), 2, 12, r)
    ss = datagen.from_strings(strs)
    chars, offs, lens = sss.to_device(ss)
    perm, lcp, _ = sss.sss_sort_batch(chars, offs, lens, first[:-1], sizes)
    sss.context().sync()
    perm, lcp = sss.u32(perm), sss.u32(lcp)
    for a, b in zip(first[:-1], first[1:]):
        sub = datagen.StringSet(ss.chars, ss.offs[a:b], ss.lens[a:b])
        want = oracle.sort(sub)
        assert np.array_equal(perm[a:b], want)
        assert np.array_equal(lcp[a:b], oracle.lcp_array(sub, want))


@pytest.mark.parametrize("seed", range(10))
def test_plain_lists_with_extensions(seed):
    """Words of 7 zeros and ones, one in twenty followed by another 0; numbers of
    seven digits of which one in twelve is another one with a 0 appended; and words
    of uneven lengths of which many are prefixes of others."""
    import paper_2404_16517_gb300 as sss
    r = np.random.default_rng(seed)
    a = [bytes((48 + r.integers(0, 2, 7)).astype(np.uint8)) + (b"0" if r.random() < 0.05 else b"") for _ in range(500)]
    b = [b"%07d" % v for v in r.integers(0, 10**7, 500)]
    for i in range(0, 500, 12):
        b[i] = b[int(r.integers(500))][:7] + b"0"
    n = int(2 ** r.uniform(6.1, 14))
    c = [bytes((97 + r.integers(0, int(r.integers(2, 4)), int(r.integers(0, 34)))).astype(np.uint8)) for _ in range(n)]
    for i in range(0, n, 3):
        c[i] = c[int(r.integers(n))] + b"a" * int(r.integers(1, 9))
    for strs in (a, b, c):
        _check(strs, (1,), _prms(sss)[:1])
