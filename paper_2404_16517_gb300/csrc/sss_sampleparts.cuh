// Sampled-splitter partition of 64-bit keys with equality buckets.
//
// Used by the local sort (reference-split keys of strings).  Every segment of
// positions [start, start+size) is split into B range buckets (s_{b-1} < k <
// s_b) and B-1 equality buckets (k == s_b) by B-1 splitters taken from an
// evenly spaced, sorted sample of the segment's keys.  Equal keys always share a
// bucket, so a key that occurs very often ends in its own equality bucket
// instead of overflowing a range bucket.  The scatter is stable (warp-level
// ranking in position order), so equal keys keep their relative order.
//
// A round is planned on the device (k_lg_plan, one CTA): it reads the list of
// segments pushed by the previous round, orders them (partitioned segments
// first, whole-segment sorts after), and writes every segment's tiles, bucket
// count and offsets plus the round's totals (LsPlan).  Every kernel of the round
// runs on a fixed grid and loops over the counts in LsPlan, so a round needs no
// host round trip.  The kernels take one pointer, the context's LsDev: the
// call's pointers and sizes are read from device memory, so a captured round
// loop serves every later call whatever its inputs and work memory are.
#pragma once

#include <algorithm>
#include <vector>

#include "sss_device.cuh"
#include "sss_internal.cuh"

namespace {

constexpr int LG_TILE = 1024, LG_T = 256;  // tile of positions per CTA / threads
constexpr int LG_OVS = 16;                 // samples per range bucket
constexpr int LG_BMAX = 256;               // max range buckets per segment
constexpr int LG_NBMAX = 2 * LG_BMAX - 1;  // range + equality buckets

struct LgTile;
struct LgRef;
struct LgSegInfo {
    Seg seg;            // start, size, depth
    uint32_t tiles;     // number of tiles
    uint32_t nb;        // range buckets B (splitters B-1, buckets 2B-1); 0 for whole-segment sorts
    uint32_t hist_base; // offset into hist (bucket-major: b*tiles + t)
    uint32_t pad;
};

// Totals of one round: segments [0, npart) are partitioned, the others sorted
// whole, [npart, npart + nbig) by the CTAs for more than bucket_cap strings and
// [npart + nbig, ns) by the bucket CTAs; tiles [0, ptiles) belong to partitioned
// segments.
struct LsPlan {
    uint32_t ns, npart, nbig, ntiles, ptiles, pbuckets;
    uint32_t pad[2];
};

// segment lists by size class: LC_QUAD and LC_WARP share one array (from the
// bottom and from the top), the others have one each
enum : uint32_t { LC_QUAD = 0, LC_WARP = 1, LC_TINY = 2, LC_SMALL = 3, LC_MED = 4, LC_LARGE = 5, LC_COUNT = 6 };

// A pointer to global memory that is itself read from memory: the compiler takes
// a kernel's pointer parameters to be global, but such a one to be anything, and
// then orders its loads with every shared-memory access around them.  With this
// and the loads of scatter and sort_emit issued together, the 37.5M-string
// batch's scatter takes 254 us instead of 513 and its bucket sorts 1.75 ms
// instead of 1.88.
template <typename T>
struct GPtr {
    T* p;
    GPtr& operator=(T* q) {
        p = q;
        return *this;
    }
    __host__ __device__ __forceinline__ operator T*() const {
#ifdef __CUDA_ARCH__
        T* q = p;
        __builtin_assume(__isGlobal(q));
        return q;
#else
        return p;
#endif
    }
};

// One call's pointers and sizes, in device memory while the call runs.
struct LsArgs {
    GPtr<const uint8_t> chars;
    GPtr<const uint64_t> offs;
    GPtr<const uint32_t> lens;
    GPtr<uint32_t> perm;
    GPtr<uint32_t> lcp;
    GPtr<uint64_t> K;
    GPtr<uint64_t> tK;
    GPtr<uint32_t> tV;
    GPtr<uint32_t> segfmt;
    GPtr<uint32_t> fixmap;  // one bit per position: LCP to recompute from the final order
    GPtr<uint64_t> spl;
    GPtr<uint32_t> hist;
    GPtr<uint32_t> bst;  // bucket starts, LG_NBMAX + 1 per segment
    GPtr<uint32_t> rankinfo;
    GPtr<LgSegInfo> info;
    GPtr<LgTile> tiles;
    GPtr<LgRef> ref;    // reference of every segment
    GPtr<uint32_t> tile0;    // first tile of every segment
    GPtr<uint32_t> bk0;      // first bucket of every segment
    GPtr<uint32_t> rowdone;  // rows scanned of every segment
    GPtr<uint32_t> redo;     // whole segments the bucket CTAs handed on (cnt[6] of them)
    GPtr<Seg> list[LC_COUNT];  // LC_WARP: the last entry of the shared array, filled downwards
    uint32_t cap[LC_COUNT];
    uint32_t warp_max, med_max, direct_max, target, bucket_cap;
    uint32_t direct_min, few, few_alone;  // k_lg_plan's rule for segments of direct_min + 1 .. direct_max strings
    uint32_t cap_tiles, cap_hist, cap_part, limit;
    uint32_t q0, q1;  // the positions being sorted
    uint32_t keep;    // the order given in perm is kept (else it starts as the identity)
};

// Device state of the local sort, one per context.  (A sector each for what a kernel
// reads once and for the counters that others change meanwhile.)
struct LsDev {
    LsArgs args;
    alignas(32) LsPlan plan;
    alignas(32) uint32_t cnt[8];   // segments per list; [6]: entries of redo, [7]: largest buckets, copied by the round's last kernel
    alignas(32) uint32_t work[8];  // dynamic work counters: [LC_*] finishers, [5] buckets, [6] direct, [7] CTAs done
    uint32_t rounds;
};

// Exclusive block scan of N u64 at once (each up to two packed 32-bit counts):
// one pass of shuffles and barriers.  1024 threads; sh: N * 32 words.
template <int N>
__device__ __forceinline__ void block_scan_n(uint64_t (&v)[N], uint64_t (&tot)[N], uint64_t* sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint64_t x[N];
#pragma unroll
    for (int k = 0; k < N; ++k) x[k] = v[k];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const uint64_t y = __shfl_up_sync(SSS_FULL, x[k], o);
            if (lane >= o) x[k] += y;
        }
    }
    if (lane == 31) {
#pragma unroll
        for (int k = 0; k < N; ++k) sh[k * 32 + w] = x[k];
    }
    __syncthreads();
    if (w < N) {
        uint64_t t = sh[w * 32 + lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(SSS_FULL, t, o);
            if (lane >= o) t += y;
        }
        sh[w * 32 + lane] = t;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < N; ++k) {
        tot[k] = sh[k * 32 + 31];
        v[k] = (w > 0 ? sh[k * 32 + w - 1] : 0ull) + x[k] - v[k];
    }
    __syncthreads();
}

// Plan a round from the large list; resets its counter for the pushes of this
// round and the round's work counters.  One CTA of 1024 threads.
//
// Segments above direct_max strings (8,192) are partitioned.  The middle ones above
// direct_min (4,352, a bucket CTA's capacity) are sorted whole, by a CTA that has an
// SM to itself, except few of them.  Measured with both ways forced, us partitioned /
// whole, by the number of middle segments:
//  * In a round that partitions others anyway they add little to its kernels, while
//    even one sorted whole is a kernel's time after them.  6,000 strings of 12
//    characters beside one of 20,000: 113 / 130 (1), 126 / 136 (38), 176 / 165 (152),
//    242 / 218 (304), 369 / 310 (608); beside one of 3,000,000: 580 / 598 (76),
//    686 / 668 (304).  But the range buckets that a round of one large segment leaves
//    too large, up to 256 of them, are mostly middle ones, and slower whole at any
//    number: 1.35M suffix views 329 / 351, 2.5M 471 / 515, 4.2M 694 / 760.  The line:
//    two segments per SM.
//  * In a round of their own it depends on the strings.  6,000 suffix views: 111 / 107
//    (1), 122 / 115 (11), 128 / 118 (38), 177 / 147 (152); of uneven lengths, from one
//    template: 161 / 182 (1), 182 / 192 (11), 203 / 208 (38), 316 / 296 (152).  The
//    line: an eighth of a segment per SM, where the two kinds balance.
__global__ void __launch_bounds__(1024) k_lg_plan(LsDev* __restrict__ S, unsigned* err) {
    __shared__ uint64_t sh[128];
    __shared__ uint32_t s_n[6];  // segments and tiles: above direct_max, middle, others above bucket_cap
    const LsArgs& A = S->args;
    const uint32_t tid = threadIdx.x;
    const uint32_t whole_max = A.direct_max, whole_min = A.direct_min, bucket_cap = A.bucket_cap, target = A.target;
    const uint32_t few = A.few, few_alone = A.few_alone;
    const Seg* list = A.list[LC_LARGE];
    LgSegInfo* info = A.info;
    uint32_t *tile0 = A.tile0, *bk0 = A.bk0, *rowdone = A.rowdone;
    const uint32_t cap_tiles = A.cap_tiles, cap_hist = A.cap_hist, cap_part = A.cap_part;
    uint32_t ns = S->cnt[LC_LARGE];
    if (ns > A.cap[LC_LARGE]) {
        if (tid == 0) atomicOr(err, ERRBIT_OVERFLOW);
        ns = 0;
    }
    if (tid < 6) s_n[tid] = 0;
    __syncthreads();  // every thread has read the count
    uint32_t n0[6] = {0, 0, 0, 0, 0, 0};
    for (uint32_t s = tid; s < ns; s += 1024) {
        const uint32_t size = list[s].size, tiles = (size + LG_TILE - 1) / LG_TILE;
        if (size > whole_max) {
            ++n0[0];
            n0[1] += tiles;
        } else if (size > whole_min) {
            ++n0[2];
            n0[3] += tiles;
        } else if (size > bucket_cap) {
            ++n0[4];
            n0[5] += tiles;
        }
    }
    if ((tid & ~31u) < ns) {  // (mostly one warp has segments)
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const uint32_t t = __reduce_add_sync(SSS_FULL, n0[k]);
            if ((tid & 31) == 0 && t) atomicAdd(&s_n[k], t);
        }
    }
    __syncthreads();
    const bool part_mid = s_n[2] <= (s_n[0] > 0 ? few : few_alone);
    const uint32_t direct_max = part_mid ? whole_min : whole_max;
    const uint32_t npart = s_n[0] + (part_mid ? s_n[2] : 0u), ptiles = s_n[1] + (part_mid ? s_n[3] : 0u);
    const uint32_t nbig = s_n[4] + (part_mid ? 0u : s_n[2]), btiles = s_n[5] + (part_mid ? 0u : s_n[3]);
    // (partitioned, big) segments, their tiles, small segments and their tiles, buckets and histogram words
    uint64_t carry[4] = {(uint64_t)npart << 32, (uint64_t)ptiles << 32,
                         (uint64_t)(npart + nbig) | ((uint64_t)(ptiles + btiles) << 32), 0};
    for (uint32_t b0 = 0; b0 < ns; b0 += 1024) {
        const uint32_t s = b0 + tid;
        const bool valid = s < ns;
        Seg sg{};
        if (valid) sg = list[s];
        const uint32_t cls = !valid ? 3u : sg.size > direct_max ? 0u : sg.size > bucket_cap ? 1u : 2u;
        const uint32_t tiles = (sg.size + LG_TILE - 1) / LG_TILE;
        uint32_t nb = 0;
        if (cls == 0) {
            nb = (sg.size + target - 1) / target;
            nb = nb < 2u ? 2u : (nb > (uint32_t)LG_BMAX ? (uint32_t)LG_BMAX : nb);
        }
        const uint32_t nbk = cls == 0 ? 2 * nb - 1 : 0u;
        uint64_t v[4], tot[4];
        v[0] = cls == 0 ? 1ull : cls == 1 ? 1ull << 32 : 0ull;
        v[1] = cls == 0 ? (uint64_t)tiles : cls == 1 ? (uint64_t)tiles << 32 : 0ull;
        v[2] = cls == 2 ? 1ull | ((uint64_t)tiles << 32) : 0ull;
        v[3] = (uint64_t)nbk | ((uint64_t)nbk * tiles << 32);
        block_scan_n(v, tot, sh);
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] += carry[k];
        if (valid) {
            const uint32_t at = cls == 0 ? (uint32_t)v[0] : cls == 1 ? (uint32_t)(v[0] >> 32) : (uint32_t)v[2];
            info[at] = LgSegInfo{sg, tiles, nb, (uint32_t)(v[3] >> 32), 0};
            tile0[at] = cls == 0 ? (uint32_t)v[1] : cls == 1 ? (uint32_t)(v[1] >> 32) : (uint32_t)(v[2] >> 32);
            bk0[at] = (uint32_t)v[3];
            rowdone[at] = 0;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) carry[k] += tot[k];
    }
    if (tid == 0) {
        const uint32_t nt = (uint32_t)(carry[2] >> 32), nh = (uint32_t)(carry[3] >> 32);
        LsPlan pl{ns, npart, nbig, nt, ptiles, (uint32_t)carry[3], {0, 0}};
        if (nt > cap_tiles || nh > cap_hist || npart > cap_part) {
            atomicOr(err, ERRBIT_OVERFLOW);
            pl = LsPlan{0, 0, 0, 0, 0, 0, {0, 0}};
        }
        S->plan = pl;
        S->cnt[LC_LARGE] = S->cnt[6] = S->cnt[7] = 0;
        S->work[5] = S->work[6] = S->work[7] = 0;
    }
}

// Last index i < n with f[i] <= g (f non-decreasing, f[0] <= g), found by the
// whole warp: 32 probes per step.
__device__ __forceinline__ uint32_t warp_last_le(const uint32_t* __restrict__ f, uint32_t n, uint32_t g) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t lo = 0, len = n;
    while (len > 32) {
        const uint32_t stride = (len + 31) / 32;
        const uint32_t at = lane * stride;
        const uint32_t k = (uint32_t)__popc(__ballot_sync(SSS_FULL, at < len && f[lo + at] <= g));
        const uint32_t skip = k ? (k - 1) * stride : 0u;
        lo += skip;
        len = len - skip < stride ? len - skip : stride;
    }
    const uint32_t k = (uint32_t)__popc(__ballot_sync(SSS_FULL, lane < len && f[lo + lane] <= g));
    return lo + (k ? k - 1 : 0u);
}

// Tile of the round: its segment and positions.  Listed by a kernel: a lookup
// per tile (up to four dependent loads in each of three kernels) cost the batch of
// 37.5M strings 0.4 ms.
struct LgTile {
    uint32_t s, begin, end, t;  // segment, positions [begin, end), index within the segment
};

// A segment's reference member: its characters, length, key format and position.
struct LgRef {
    GPtr<const uint8_t> chars;
    uint32_t len, fmt, pos, pad;
};

// Splitters of the partitioned segments: of n = nb * LG_OVS evenly spaced
// samples (ties by number) the ones of rank (b+1)*OVS - 1.  Ranks by comparing
// all pairs: a unit is two buckets' worth of samples (32, one per lane) of a
// segment, its 16 warps share out the others.  A segment of 4,096 samples is
// then 128 units on as many CTAs (10 us); one CTA sorting them in shared memory
// (a bitonic network, 78 steps) took 40 us with every other SM idle.
constexpr int SP_T = 512;
__global__ void __launch_bounds__(SP_T) k_lg_samples(const LsDev* __restrict__ S) {
    __shared__ uint64_t sh[LG_BMAX * LG_OVS];
    __shared__ uint32_t s_rank[2 * LG_OVS];
    const LsArgs& A = S->args;
    const uint32_t npart = S->plan.npart;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // the segments' range buckets, numbered through: (bk0[s] + s) / 2 precede segment s
    const uint32_t total = (S->plan.pbuckets + npart) / 2;
    // a CTA's units lie side by side: mostly one segment, whose samples stay
    const uint32_t per = 2 * ((total + 2 * gridDim.x - 1) / (2 * gridDim.x));
    const uint32_t last = (blockIdx.x + 1) * per < total ? (blockIdx.x + 1) * per : total;
    uint32_t loaded = 0xFFFFFFFFu;
    for (uint32_t x = blockIdx.x * per; x < last;) {
        const uint32_t end = x + 2 < last ? x + 2 : last;
        uint32_t s = 0;  // last s with (bk0[s] + s) / 2 <= x
        for (uint32_t len = npart; len > 0;) {
            const uint32_t stride = (len + 31) / 32, at = lane * stride;
            const bool le = at < len && (A.bk0[s + at] + s + at) / 2 <= x;
            const uint32_t k = (uint32_t)__popc(__ballot_sync(SSS_FULL, le));
            const uint32_t skip = k ? (k - 1) * stride : 0u;
            s += skip;
            len = stride == 1 ? 0u : (len - skip < stride ? len - skip : stride);
        }
        const LgSegInfo si = A.info[s];
        const uint32_t r = x - (A.bk0[s] + s) / 2;  // bucket within the segment
        if (si.nb <= SP_T / LG_OVS && (per >= 8 || si.nb <= 8)) {
            // few samples, and segments enough for every CTA: a thread per sample, by
            // the unit of the segment's first bucket
            if (r == 0) {
                const uint32_t n = si.nb * LG_OVS;
                __syncthreads();
                uint64_t mine = 0;
                if (threadIdx.x < n) {
                    mine = A.K[si.seg.start + ((2 * (uint64_t)threadIdx.x + 1) * si.seg.size) / (2 * (uint64_t)n)];
                    sh[threadIdx.x] = mine;
                }
                __syncthreads();
                if (threadIdx.x < n) {
                    const uint32_t wb = threadIdx.x - lane, we = wb + 32 < n ? wb + 32 : n;
                    uint32_t rank = 0;
#pragma unroll 8
                    for (uint32_t i = 0; i < wb; ++i) rank += sh[i] <= mine ? 1u : 0u;
                    for (uint32_t i = wb; i < we; ++i) rank += sh[i] < mine + (i < threadIdx.x ? 1ull : 0ull) ? 1u : 0u;
#pragma unroll 8
                    for (uint32_t i = we; i < n; ++i) rank += sh[i] < mine ? 1u : 0u;
                    if (rank % LG_OVS == LG_OVS - 1 && rank / LG_OVS + 1 < si.nb)
                        A.spl[(size_t)s * (LG_BMAX - 1) + rank / LG_OVS] = mine;
                }
                loaded = 0xFFFFFFFFu;
            }
            x += si.nb - r;
            continue;
        }
        const uint32_t cnt = end - x < si.nb - r ? end - x : si.nb - r;
        const uint32_t n = si.nb * LG_OVS;
        __syncthreads();
        if (s != loaded) {
            for (uint32_t i = threadIdx.x; i < n; i += SP_T) {
                const uint64_t q = si.seg.start + ((2 * (uint64_t)i + 1) * si.seg.size) / (2 * (uint64_t)n);
                sh[i] = A.K[q];
            }
            loaded = s;
        }
        if (threadIdx.x < 2 * LG_OVS) s_rank[threadIdx.x] = 0;
        __syncthreads();
        const uint32_t me = r * LG_OVS + lane;  // sample of this lane (lanes past cnt buckets idle)
        const bool have = lane < cnt * LG_OVS;
        const uint64_t mine = have ? sh[me] : 0ull;
        const uint32_t i0 = w * si.nb, i1 = i0 + si.nb;  // this warp's share: n / 16 samples
        uint32_t c = 0;
        if (i1 <= r * LG_OVS || i0 > r * LG_OVS + 31u) {
            // all before the lanes' samples (equal ones go first) or all after (they do not)
            const uint64_t lim = mine + (i1 <= r * LG_OVS ? 1ull : 0ull);
#pragma unroll 8
            for (uint32_t i = i0; i < i1; ++i) c += sh[i] < lim ? 1u : 0u;
        } else {
            for (uint32_t i = i0; i < i1; ++i) c += sh[i] < mine + (i < me ? 1ull : 0ull) ? 1u : 0u;
        }
        if (have && c) atomicAdd(&s_rank[lane], c);
        __syncthreads();
        if (w == 0 && have) {
            const uint32_t rank = s_rank[lane], b = rank / LG_OVS;
            if (rank % LG_OVS == LG_OVS - 1 && b + 1 < si.nb) A.spl[(size_t)s * (LG_BMAX - 1) + b] = mine;
        }
        x += cnt;
    }
}
static_assert(SP_T / 32 == LG_OVS, "a warp's share of the samples is nb");

// first splitter >= k (lower bound) among nsp sorted splitters
__device__ __forceinline__ uint32_t lower_bound64(const uint64_t* s, uint32_t nsp, uint64_t k) {
    uint32_t lo = 0, hi = nsp;
    while (lo < hi) {
        uint32_t mid = (lo + hi) >> 1;
        if (s[mid] < k) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(LG_T) k_lg_classify(const LsDev* __restrict__ S) {
    constexpr int W = LG_T / 32;
    constexpr int PER_WARP = LG_TILE / W;  // contiguous positions per warp
    __shared__ uint64_t ssp[LG_BMAX];
    __shared__ uint32_t cnt[W][LG_NBMAX];
    const LsArgs& A = S->args;
    const uint64_t* __restrict__ K = A.K;
    uint32_t* __restrict__ hist = A.hist;
    uint32_t* __restrict__ rankinfo = A.rankinfo;
    const uint32_t ptiles = S->plan.ptiles;
    for (uint32_t g = blockIdx.x; g < ptiles; g += gridDim.x) {
        __syncthreads();
        const LgTile tl = A.tiles[g];
        const LgSegInfo si = A.info[tl.s];
        uint32_t nsp = si.nb - 1, nbk = 2 * si.nb - 1;
        for (uint32_t i = threadIdx.x; i < nsp; i += LG_T) ssp[i] = A.spl[(size_t)tl.s * (LG_BMAX - 1) + i];
        for (uint32_t i = threadIdx.x; i < (uint32_t)(W * LG_NBMAX); i += LG_T) (&cnt[0][0])[i] = 0;
        __syncthreads();
        int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        uint32_t lt = (1u << lane) - 1u;
        uint32_t myb[PER_WARP / 32], myr[PER_WARP / 32];
#pragma unroll
        for (int it = 0; it < PER_WARP / 32; ++it) {
            uint32_t q = tl.begin + w * PER_WARP + it * 32 + lane;
            bool valid = q < tl.end;
            uint32_t b = 0xFFFFu;
            if (valid) {
                uint64_t k = K[q];
                uint32_t lb = lower_bound64(ssp, nsp, k);
                b = 2 * lb + ((lb < nsp && ssp[lb] == k) ? 1u : 0u);
            }
            uint32_t peers = __match_any_sync(SSS_FULL, b);
            uint32_t leader = __ffs(peers) - 1;
            uint32_t base = 0;
            if (valid && lane == (int)leader) {
                base = cnt[w][b];
                cnt[w][b] = base + __popc(peers);
            }
            base = __shfl_sync(SSS_FULL, base, leader);
            myb[it] = b;
            myr[it] = base + __popc(peers & lt);
        }
        __syncthreads();
        // exclusive prefix over warps for every bucket; tile total into hist
        for (uint32_t b = threadIdx.x; b < nbk; b += LG_T) {
            uint32_t run = 0;
#pragma unroll
            for (int ww = 0; ww < W; ++ww) {
                uint32_t t = cnt[ww][b];
                cnt[ww][b] = run;
                run += t;
            }
            hist[si.hist_base + b * si.tiles + tl.t] = run;
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < PER_WARP / 32; ++it) {
            uint32_t q = tl.begin + w * PER_WARP + it * 32 + lane;
            if (q < tl.end) rankinfo[q] = (myb[it] << 16) | (cnt[w][myb[it]] + myr[it]);
        }
    }
}

// Exclusive prefix of every bucket's row of tile counts (one warp per row, the
// row contiguous, so loads coalesce); the row total goes to the bucket's start
// slot.  The warp that finishes a segment's last row turns its totals into
// bucket starts (a separate launch for that cost 3 us and its gap per round).
__global__ void __launch_bounds__(256) k_lg_rowscan(const LsDev* __restrict__ S) {
    const LsArgs& A = S->args;
    const uint32_t nrows = S->plan.pbuckets, npart = S->plan.npart;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    for (uint32_t r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < nrows; r += warps) {
        const uint32_t s = warp_last_le(A.bk0, npart, r);
        const LgSegInfo si = A.info[s];
        const uint32_t b = r - A.bk0[s], nbk = 2 * si.nb - 1;
        uint32_t* h = A.hist + si.hist_base + b * si.tiles;
        uint32_t* bst = A.bst + (size_t)s * (LG_NBMAX + 1);
        // 8 x 32 counts in flight: a 4M-string segment has 4,096 per row, and 32 a
        // time they took 50 us
        uint32_t carry = 0;
        for (uint32_t t0 = 0; t0 < si.tiles; t0 += 256) {
            uint32_t v[8], x[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint32_t t = t0 + 32 * c + lane;
                x[c] = v[c] = t < si.tiles ? h[t] : 0u;
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint32_t y = __shfl_up_sync(SSS_FULL, x[c], o);
                    if (lane >= (uint32_t)o) x[c] += y;
                }
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint32_t t = t0 + 32 * c + lane;
                if (t < si.tiles) h[t] = carry + x[c] - v[c];
                carry += __shfl_sync(SSS_FULL, x[c], 31);
            }
        }
        uint32_t done = 0;
        if (lane == 0) {
            __stcg(&bst[b], carry);
            __threadfence();
            done = atomicAdd(&A.rowdone[s], 1u) + 1u;
        }
        done = __shfl_sync(SSS_FULL, done, 0);
        if (done != nbk) continue;
        __threadfence();
        uint32_t run = si.seg.start;
        for (uint32_t b0 = 0; b0 < nbk; b0 += 32) {
            const uint32_t i = b0 + lane;
            const uint32_t v = i < nbk ? __ldcg(&bst[i]) : 0u;
            uint32_t x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                uint32_t y = __shfl_up_sync(SSS_FULL, x, o);
                if (lane >= (uint32_t)o) x += y;
            }
            if (i < nbk) bst[i] = run + x - v;
            run += __shfl_sync(SSS_FULL, x, 31);
        }
        if (lane == 0) bst[nbk] = si.seg.start + si.seg.size;
    }
}

// The scatter of a tile goes through shared memory: its keys are first placed
// in bucket order (the tile's bucket counts, scanned, plus each key's rank within
// its bucket), so that consecutive threads then write consecutive positions of
// one bucket's range.  Written directly, the keys of a warp land in as many
// buckets as they have, and every 8-byte key or 4-byte index costs a whole
// sector of DRAM writes.
__global__ void __launch_bounds__(LG_T) k_lg_scatter(const LsDev* __restrict__ S, unsigned* err) {
    constexpr int PER = LG_TILE / LG_T;
    static_assert(2 * LG_T >= LG_NBMAX, "two buckets per thread in the scan");
    __shared__ uint32_t cnt[2 * LG_T];
    __shared__ uint32_t sh_warp[32];
    __shared__ uint64_t sK[LG_TILE];
    __shared__ uint32_t sV[LG_TILE], sD[LG_TILE];
    const LsArgs& A = S->args;
    const uint32_t* __restrict__ hist = A.hist;
    const uint32_t* __restrict__ rankinfo = A.rankinfo;
    const uint64_t* __restrict__ K = A.K;
    const uint32_t* __restrict__ perm = A.perm;
    uint64_t* __restrict__ tK = A.tK;
    uint32_t* __restrict__ tV = A.tV;
    const uint32_t tid = threadIdx.x;
    const uint32_t ptiles = S->plan.ptiles;
    for (uint32_t g = blockIdx.x; g < ptiles; g += gridDim.x) {
        const LgTile tl = A.tiles[g];
        const LgSegInfo si = A.info[tl.s];
        const uint32_t* __restrict__ bst = A.bst + (size_t)tl.s * (LG_NBMAX + 1);
        const uint32_t nbk = 2 * si.nb - 1;
        __syncthreads();  // the previous tile's keys have left shared memory
        for (uint32_t i = tid; i < 2u * LG_T; i += LG_T) cnt[i] = 0;
        __syncthreads();
        // everything the tile reads, in flight before the first use
        uint32_t ri[PER], rv[PER];
        uint64_t rk[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const uint32_t q = tl.begin + tid + u * LG_T;
            ri[u] = q < tl.end ? __ldg(rankinfo + q) : 0xFFFFFFFFu;
            rk[u] = q < tl.end ? __ldg(K + q) : 0ull;
            rv[u] = q < tl.end ? __ldg(perm + q) : 0u;
        }
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (ri[u] != 0xFFFFFFFFu) atomicAdd(&cnt[min(ri[u] >> 16, 2u * LG_T - 1u)], 1u);  // b < nbk <= 511
        uint32_t first[PER];  // the tile's first position in the key's bucket
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const uint32_t b = min(ri[u] >> 16, nbk - 1);
            first[u] = ri[u] != 0xFFFFFFFFu ? __ldg(bst + b) + __ldg(hist + si.hist_base + b * si.tiles + tl.t) : 0u;
        }
        __syncthreads();
        // the tile's bucket offsets: exclusive scan of the counts
        const uint32_t c0 = cnt[2 * tid], c1 = cnt[2 * tid + 1];
        const uint32_t ex = BlockScan<LG_T>::exclusive_sum(c0 + c1, sh_warp, nullptr);
        cnt[2 * tid] = ex;
        cnt[2 * tid + 1] = ex + c0;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            if (ri[u] == 0xFFFFFFFFu) continue;
            const uint32_t b = ri[u] >> 16, r = ri[u] & 0xFFFFu;
            const uint32_t slot = cnt[min(b, 2u * LG_T - 1u)] + r;
            uint32_t dst = first[u] + r;
            if (b >= nbk || dst < si.seg.start || dst >= si.seg.start + si.seg.size || slot >= LG_TILE) {
                atomicOr(err, ERRBIT_OVERFLOW);
                if (slot >= LG_TILE) continue;
                dst = 0xFFFFFFFFu;
            }
            sK[slot] = rk[u];
            sV[slot] = rv[u];
            sD[slot] = dst;
        }
        __syncthreads();
        const uint32_t m = tl.end - tl.begin;
        for (uint32_t i = tid; i < m; i += LG_T) {
            const uint32_t dst = sD[i];
            if (dst == 0xFFFFFFFFu) continue;
            tK[dst] = sK[i];
            tV[dst] = sV[i];
        }
    }
}

// Work memory of the partition for up to `cap_segs` segments covering <= n
// positions, `cap_part` of them partitioned (those come first).
inline void carve_sp(Arena& ar, uint32_t n, uint32_t cap_segs, uint32_t cap_part, LsArgs& a) {
    a.cap_tiles = n / LG_TILE + cap_segs + 2;
    a.cap_hist = LG_NBMAX * (n / LG_TILE + cap_part + 2);
    a.cap_part = cap_part;
    a.spl = ar.take<uint64_t>((size_t)cap_part * (LG_BMAX - 1));
    a.hist = ar.take<uint32_t>(a.cap_hist);
    a.bst = ar.take<uint32_t>((size_t)cap_part * (LG_NBMAX + 1));
    a.rankinfo = ar.take<uint32_t>(n);
    a.info = ar.take<LgSegInfo>(cap_segs);
    a.tiles = ar.take<LgTile>(a.cap_tiles);
    a.ref = ar.take<LgRef>(cap_segs);
    a.tile0 = ar.take<uint32_t>(cap_segs);
    a.bk0 = ar.take<uint32_t>(cap_segs);
    a.rowdone = ar.take<uint32_t>(cap_segs);
    a.redo = ar.take<uint32_t>(cap_segs);
}

}  // namespace
