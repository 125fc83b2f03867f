"""Performance cases of the string sorter: what its users have it sort, through
the package's own calls.

Inputs follow the shapes of the repository's workloads (template sets, requests
of strings of uneven length, suffix views of a Markov text, the length-skewed
set, packed instances), drawn with torch on the GPU from the seed alone.  The
sizes of a batch's instances are the quantiles of their distribution, shuffled
by the seed, so that a case's work does not depend on the seed.

Outputs are whole numbers (orders, LCP arrays, distinguishing prefixes) and
therefore equal on any two correct runs; no 64-bit reference values are needed.
"""
from __future__ import annotations

import math
import random
import statistics

import torch

import paper_2404_16517_gb300 as sss

DEV = "cuda"
CHUNK = 1 << 18  # strings per generation step of the uneven sets


# --------------------------------------------------------------------------
# cases

def _template(n, length, templates, shared):
    """n strings of one length over A-Z; the first `shared` characters come from
    one of `templates` templates."""
    return dict(set="template", n=n, length=length, templates=templates, shared=shared)


def _uneven(n, len_lo, len_hi, sigma, ratio):
    """n strings with lengths uniform in len_lo..len_hi over sigma letters; a
    string copies about ratio of its length from one template."""
    return dict(set="uneven", n=n, len_lo=len_lo, len_hi=len_hi, sigma=sigma, ratio=ratio)


def _views(text, n, max_len):
    """n suffixes of a Markov text, cut at max_len characters (views)."""
    return dict(set="views", text=text, n=n, max_len=max_len)


def _skew(n, short, long):
    """n strings over A-Z, short ones, and long ones (those starting with Z)
    that share all but their last characters."""
    return dict(set="skew", n=n, short=short, long=long)


def listed():
    return [
        # the smallest use: one short list sorted by a program that waits for it
        dict(name="sort_1000", kind="sort", p=1, dist=False, chars=False, **_uneven(1000, 8, 64, 26, 0.5)),
        # the plain one-partition sort, with distinguishing prefixes
        dict(name="sort_65536x100", kind="sort", p=1, dist=True, chars=False, **_template(65536, 100, 4, 42)),
        # one request of a serving stream alone: uneven lengths up to 1000
        dict(name="sort_300007", kind="sort", p=1, dist=False, chars=False, **_uneven(300007, 16, 1000, 26, 0.6)),
        # the whole merge sort with few partitions
        dict(name="pdms_1m_p4", kind="sort", p=4, dist=False, chars=False, **_template(1 << 20, 500, 64, 242)),
        # the headline workload: 4.19M strings of 500 characters, 16 partitions
        dict(name="pdms_4m_p16", kind="sort", p=16, dist=False, chars=False, **_template(1 << 22, 500, 64, 242)),
        # many partitions of overlapping views with long shared prefixes, with dist
        dict(name="pdms_views_p64", kind="sort", p=64, dist=True, chars=False, **_views(1 << 22, 1 << 21, 256)),
        # short strings with a skewed share of long ones, character-based sampling
        dict(name="pdms_skew_p16", kind="sort", p=16, dist=False, chars=True, **_skew(1 << 22, 20, 1000)),
        # thousands of independent instances in one graph launch
        dict(name="batch_4096", kind="batch", m=4096, sizes="loguniform", lo=6.0, hi=16.0, graph=True, len_lo=8,
             len_hi=300, sigma=4),
        # what one step of the request server sorts: about eleven requests at once
        dict(name="batch_serve_11", kind="batch", m=11, sizes="lognormal", lo=14.0, hi=1.5, graph=False, len_lo=16,
             len_hi=1000, sigma=26),
        # suffix array and LCP array of a text with short repeats
        dict(name="text_4m", kind="text", n=1 << 22, copies=0, longest=0),
        # and of an odd-sized one in which passages occur again (rank doubling)
        dict(name="text_repeats_1m", kind="text", n=1000003, copies=200, longest=4096),
        # strings that start in host memory: upload, sort, results back
        dict(name="host_1m_p16", kind="host", p=16, **_template(1 << 20, 500, 64, 242)),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sort", "sort", "pdms", "pdms", "batch", "batch", "text", "host"])
    if kind in ("sort", "pdms"):
        p = 1 if kind == "sort" else rng.choice([2, 3, 4, 7, 16, 16, 31, 64, 128])
        shape = rng.choice(["template", "template", "uneven", "uneven", "views", "skew"])
        n = _log(rng, 1000 if p == 1 else 20000, 1 << 22)
        if shape == "template":
            length = rng.choice([64, 100, 101, 250, 500])
            s = _template(n, length, rng.choice([1, 4, 64, 100]), int(length * rng.uniform(0.1, 0.7)))
        elif shape == "uneven":
            hi = rng.choice([64, 300, 1000])
            n = min(n, (1 << 31) // hi)
            s = _uneven(n, rng.choice([1, 8, 16]), hi, rng.choice([4, 26]), round(rng.uniform(0.1, 0.9), 3))
        elif shape == "views":
            n = min(n, 1 << 21)
            s = _views(max(4096, 2 * n), n, rng.choice([64, 255, 256]))
        else:
            s = _skew(n, rng.choice([12, 20, 33]), rng.choice([200, 1000]))
        return dict(kind="sort", p=p, dist=rng.random() < 0.5, chars=p > 1 and rng.random() < 0.25, **s)
    if kind == "batch":
        if rng.random() < 0.5:
            return dict(kind="batch", m=_log(rng, 16, 4000), sizes="loguniform", lo=rng.choice([4.0, 6.0]),
                        hi=rng.choice([10.0, 13.0, 16.0]), graph=rng.random() < 0.5, len_lo=8, len_hi=300, sigma=4)
        return dict(kind="batch", m=_log(rng, 1, 64), sizes="lognormal", lo=round(rng.uniform(11.0, 14.0), 2), hi=1.5,
                    graph=rng.random() < 0.25, len_lo=16, len_hi=1000, sigma=26)
    if kind == "text":
        n = _log(rng, 2000, 1 << 22)
        if rng.random() < 0.5:
            return dict(kind="text", n=n, copies=0, longest=0)
        n = min(n, 1 << 20)
        return dict(kind="text", n=n, copies=rng.choice([1, 20, 200]), longest=min(n // 4, rng.choice([256, 2048, 4096])))
    return dict(kind="host", p=rng.choice([1, 4, 16]),
                **_template(_log(rng, 20000, 1 << 20), rng.choice([100, 500]), 64, rng.choice([40, 60])))


# --------------------------------------------------------------------------
# inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _letters(g, count, sigma):
    """count uniform letters of A-Z, or of ACGT for sigma = 4."""
    out = torch.empty(count, dtype=torch.uint8, device=DEV)
    for a in range(0, count, 1 << 29):
        part = out[a:a + (1 << 29)]
        part.random_(0, sigma, generator=g)
        if sigma != 4:
            part += 65
    if sigma == 4:
        acgt = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=DEV)
        for a in range(0, count, 1 << 27):
            part = out[a:a + (1 << 27)]
            part.copy_(acgt[part.to(torch.int32)])
    return out


def _offsets(lens):
    offs = torch.zeros(lens.numel(), dtype=torch.int64, device=DEV)
    if lens.numel() > 1:
        torch.cumsum(lens[:-1], 0, dtype=torch.int64, out=offs[1:])
    return offs


def _template_set(c, g):
    n, length, shared = c["n"], c["length"], c["shared"]
    tmpl = _letters(g, c["templates"] * length, 26).view(-1, length)
    pick = torch.randint(0, c["templates"], (n,), generator=g, device=DEV)
    chars = _letters(g, n * length, 26)
    rows = chars.view(n, length)
    for a in range(0, n, 1 << 20):
        rows[a:a + (1 << 20), :shared] = tmpl[pick[a:a + (1 << 20)], :shared]
    offs = torch.arange(n, dtype=torch.int64, device=DEV) * length
    return chars, offs, torch.full((n,), length, dtype=torch.int32, device=DEV)


def _instances(g, sizes, ratios, len_lo, len_hi, sigma):
    """Strings of instance k copy max(0, round(ratio * length) - log_sigma(size) - 1)
    characters of its template; the rest is uniform."""
    m, n = len(sizes), sum(sizes)
    lens = torch.randint(len_lo, len_hi + 1, (n,), generator=g, device=DEV, dtype=torch.int32)
    offs = _offsets(lens)
    sz = torch.tensor(sizes, device=DEV)
    inst = torch.repeat_interleave(torch.arange(m, device=DEV), sz)
    own = torch.tensor([math.ceil(math.log(max(s, 2)) / math.log(sigma)) + 1 for s in sizes], device=DEV)
    cp = (torch.tensor(ratios, device=DEV)[inst] * lens).round().long().sub_(own[inst]).clamp_(min=0)
    chars = _letters(g, int(lens.sum(dtype=torch.int64)), sigma)
    tmpl = _letters(g, m * len_hi, sigma)
    for a in range(0, n, CHUNK):
        b = min(n, a + CHUNK)
        part = cp[a:b]
        owner = torch.repeat_interleave(torch.arange(b - a, device=DEV), part)
        at = torch.arange(owner.numel(), device=DEV) - (torch.cumsum(part, 0) - part)[owner]
        chars[offs[a:b][owner] + at] = tmpl[inst[a:b][owner] * len_hi + at]
    return chars, offs, lens


def _markov(g, n, sigma=64):
    """A text of n characters: order-2 Markov chains over sigma symbols, 4096 of
    them side by side, with sparse random transition rows."""
    k = torch.empty(sigma * sigma, sigma, device=DEV)
    # exponents of uniforms: most of a row's weight falls on a few symbols
    k.uniform_(generator=g).pow_(10.0).clamp_(min=1e-12)
    cdf = torch.cumsum(k / k.sum(1, keepdim=True), 1)
    cdf[:, -1] = 1.0
    chains = min(4096, max(1, n // 64))
    steps = -(-n // chains)
    out = torch.empty(steps, chains, dtype=torch.uint8, device=DEV)
    a = torch.randint(0, sigma, (chains,), generator=g, device=DEV)
    b = torch.randint(0, sigma, (chains,), generator=g, device=DEV)
    u = torch.rand(steps, chains, 1, generator=g, device=DEV)
    for t in range(steps):
        nxt = torch.searchsorted(cdf[a * sigma + b], u[t]).squeeze(1).clamp_(max=sigma - 1)
        out[t] = nxt
        a, b = b, nxt
    return (out + 0x21).t().reshape(-1)[:n].contiguous()


def _text(c, seed, g):
    t = _markov(g, c["n"])
    r = random.Random(seed)
    for _ in range(c["copies"]):
        length = _log(r, 64, max(65, c["longest"]))
        src, dst = r.randrange(c["n"] - length), r.randrange(c["n"] - length)
        t[dst:dst + length] = t[src:src + length].clone()
    return t


def _strings(c, seed):
    g = _gen(seed)
    if c["set"] == "template":
        return _template_set(c, g)
    if c["set"] == "uneven":
        return _instances(g, [c["n"]], [c["ratio"]], c["len_lo"], c["len_hi"], c["sigma"])
    if c["set"] == "views":
        text = _markov(g, c["text"])
        offs = torch.randperm(c["text"], generator=g, device=DEV)[:c["n"]].contiguous()
        return text, offs, (c["text"] - offs).clamp(max=c["max_len"]).to(torch.int32)
    first = torch.randint(0, 26, (c["n"],), generator=g, device=DEV)
    lens = torch.where(first == 25, c["long"], c["short"]).to(torch.int32)
    offs = _offsets(lens)
    chars = _letters(g, int(lens.sum(dtype=torch.int64)), 26)
    tmpl = _letters(g, c["long"], 26)
    at = offs[first == 25]
    for a in range(0, at.numel(), 1 << 16):
        part = at[a:a + (1 << 16), None] + torch.arange(1, c["long"] - 8, device=DEV)[None, :]
        chars[part] = tmpl[1:c["long"] - 8].expand(part.shape)
    chars[offs] = (first + 65).to(torch.uint8)
    return chars, offs, lens


def _batch_sizes(c):
    m = c["m"]
    if c["sizes"] == "loguniform":
        return [int(2.0 ** (c["lo"] + (c["hi"] - c["lo"]) * (k + 0.5) / m)) for k in range(m)]
    z = statistics.NormalDist()
    return [max(1, round(2.0 ** c["lo"] * math.exp(c["hi"] * z.inv_cdf((k + 0.5) / m)))) for k in range(m)]


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _u32(n):
    return torch.empty(n, dtype=torch.int32, device=DEV)


def prepare(case, seed):
    c = case
    if c["kind"] == "text":
        return dict(kind="text", text=_text(c, seed, _gen(seed)), sa=_u32(c["n"]), lcp=_u32(c["n"]))
    if c["kind"] == "batch":
        r = random.Random(seed)
        sizes = _batch_sizes(c)
        r.shuffle(sizes)
        ratios = [0.1 + 0.8 * (k + 0.5) / c["m"] for k in range(c["m"])]
        r.shuffle(ratios)
        chars, offs, lens = _instances(_gen(seed), sizes, ratios, c["len_lo"], c["len_hi"], c["sigma"])
        first = [0]
        for s in sizes[:-1]:
            first.append(first[-1] + s)
        n = lens.numel()
        return dict(kind="batch", s=(chars, offs, lens), first=first, sizes=sizes,
                    prm=sss.params(flags=sss.SSS_FLAG_GRAPH if c["graph"] else 0), perm=_u32(n), lcp=_u32(n))
    s = _strings(c, seed)
    n = c["n"]
    if c["kind"] == "host":
        h = tuple(_pinned(t) for t in s)
        return dict(kind="host", h=h, d=tuple(torch.empty_like(t) for t in s), p=c["p"], perm=_u32(n), lcp=_u32(n),
                    h_perm=_pinned(torch.zeros(n, dtype=torch.int32)),
                    h_lcp=_pinned(torch.zeros(n, dtype=torch.int32)))
    return dict(kind="sort", s=s, p=c["p"], prm=sss.params(flags=sss.SSS_FLAG_CHAR_SAMPLING if c["chars"] else 0),
                perm=_u32(n), lcp=_u32(n), dist=_u32(n) if c["dist"] else None)


# --------------------------------------------------------------------------
# one pass

def run(state):
    t = state
    if t["kind"] == "sort":
        perm, lcp, dist, _ = sss.sss_sort(*t["s"], t["p"], t["prm"], t["perm"], t["lcp"], out_dist=t["dist"])
        return [perm, lcp] if dist is None else [perm, lcp, dist]
    if t["kind"] == "batch":
        perm, lcp, _ = sss.sss_sort_batch(*t["s"], t["first"], t["sizes"], t["prm"], t["perm"], t["lcp"])
        return [perm, lcp]
    if t["kind"] == "text":
        return list(sss.sss_suffix_sort(t["text"], out_sa=t["sa"], out_lcp=t["lcp"]))
    perm, lcp = sss.sss_sort_host(*t["h"], t["p"], *t["d"], out_perm=t["perm"], out_lcp=t["lcp"],
                                  h_out_perm=t["h_perm"], h_out_lcp=t["h_lcp"])
    return [perm, lcp, t["h_perm"], t["h_lcp"]]


# --------------------------------------------------------------------------
# what a pass cannot do without

def _log_base(n, sigma):
    return math.log(max(n, 2)) / math.log(sigma)


def _needed_chars(c):
    """Characters that decide the order (about the sum of the distinguishing
    prefixes): a shared prefix, then as many as tell its sharers apart."""
    n = c["n"]
    if c["set"] == "template":
        return n * min(c["length"], c["shared"] + _log_base(n / c["templates"], 26) + 1)
    if c["set"] == "uneven":
        mean = (c["len_lo"] + c["len_hi"]) / 2
        return n * min(mean, max(0.0, c["ratio"] * mean - _log_base(n, c["sigma"]) - 1) + _log_base(n, c["sigma"]) + 1)
    if c["set"] == "views":
        return n * min(c["max_len"], _log_base(n, 8) + 1)
    return n * (25 / 26 * min(c["short"], _log_base(n, 26) + 1) + c["long"] / 26)


def work(case):
    c = case
    if c["kind"] == "text":  # the text once, both arrays once
        return {"bytes": 9.0 * c["n"], "flops": 0}
    if c["kind"] == "batch":
        n = sum(_batch_sizes(c))
        return {"bytes": n * (0.5 * (c["len_lo"] + c["len_hi"]) / 2 + 20.0), "flops": 0}
    n = c["n"]
    if c["kind"] == "host":  # every character crosses the link
        return {"bytes": n * (c["length"] + 12.0 + 8.0) + _needed_chars(c) + 20.0 * n, "flops": 0}
    # the views (12 bytes each) and both outputs, and dist
    return {"bytes": _needed_chars(c) + n * (20.0 + (4.0 if c["dist"] else 0.0)), "flops": 0}
