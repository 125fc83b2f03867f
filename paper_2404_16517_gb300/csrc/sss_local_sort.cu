// Stage A: local string sort of every partition with LCP-array output
// (Section 3, "Initialization": each PE sorts its local strings; the LCP array
// is a by-product of sorting).  A6: exact distinguishing prefixes (Section 2).
//
// Design (GB300): MSD radix sort with reference-split keys.
//  * A segment is a run of positions whose strings share their first `depth`
//    characters.  Every member is compared with one of them (the reference, a
//    long one of a few candidates) from `depth` on: its full LCP v with the
//    reference, its next characters and which side of the reference it falls on
//    make a 64-bit key (ref_key in sss_device.cuh) whose order is string order on
//    the first depth + v + C characters (C = 4..6, by the reference's length).
//    Each member thus skips its own shared prefix with the reference; a plain
//    common-prefix skip would only advance the whole segment by the smallest v.
//  * Segments of more than cta_cap strings take multi-CTA rounds: compute the
//    keys, then either sort the whole segment in one CTA's shared memory (up to
//    direct_cap strings) or sample splitters, classify into range and equality
//    buckets (equal keys always share a bucket), scatter stably and sort each
//    range bucket in shared memory; groups of equal keys become new segments.
//  * All the others, the call's own and those that the rounds leave, are finished
//    once after the last round, inside one CTA, warp or four lanes each: keys are
//    gathered, sorted as (group, key, index) and split, until every group is a
//    single string or a run of equal strings.
//  * Rounds, finishers and seams are one graph launch that reads everything of
//    the call from device memory (LsDev).
//  * LCP values fall out at every split (key_lcp); equal strings get lcp = their
//    length.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "sss_device.cuh"
#include "sss_internal.cuh"
#include "sss_sampleparts.cuh"

namespace {

constexpr uint32_t DONE = 0xFFFFFFFFu;

// size classes
constexpr int WF_WARPS = 8;                     // group finishers: warps per CTA
constexpr int QUAD_W = 4;                       // segments of <= 4 strings: 4 lanes each, 8 per warp
constexpr int TINY_T = 64, TINY_CAP = 64;       // segments of warp_cap+1 .. 64 strings
constexpr int SM_T = 128, SM_CAP = 512;         // segments of 65 .. 512 strings
constexpr int MED_T = 512, MED_CAP = 2048;      // segments of 513 .. cta_cap (<= 2048) strings, 2 CTAs per SM
constexpr int BK_T = 512, BK_CAP = 4352;        // bucket sort CTA (bucket targets above BKS_CAP / 2)
constexpr int BKS_T = 256, BKS_CAP = 2048;      // bucket sort CTA for targets <= BKS_CAP / 2 (4 CTAs per SM)
constexpr int DIRECT_T = 1024, DIRECT_CAP = 8192;  // whole-segment sort CTA (segments <= direct_cap)

// size class of a segment of >= 2 strings: quad <= QUAD_W, warp <= warp_max <
// tiny <= TINY_CAP < small <= SM_CAP < med <= med_max < large
__device__ __forceinline__ uint32_t seg_class(const LsArgs& A, uint32_t size) {
    if (size <= A.warp_max) return size <= (uint32_t)QUAD_W ? LC_QUAD : LC_WARP;
    if (size <= (uint32_t)TINY_CAP) return LC_TINY;
    if (size <= A.med_max) return size <= (uint32_t)SM_CAP ? LC_SMALL : LC_MED;
    return LC_LARGE;
}

// Entry i of list c.  The two short classes share one array, quad from the
// bottom and warp from the top; they never meet, as the segments on the short
// lists are disjoint over all rounds (a short segment is final: its positions
// never return to the large list) and hold >= 2 strings each.
__device__ __forceinline__ void put_seg(const LsArgs& A, uint32_t c, uint32_t i, const Seg& sg, unsigned* err) {
    if (i >= A.cap[c]) {
        atomicOr(err, ERRBIT_OVERFLOW);
        return;
    }
    Seg* at = A.list[c];
    if (c == LC_WARP) at -= i;
    else at += i;
    *at = sg;
}

__device__ __forceinline__ void push_seg(const LsArgs& A, uint32_t* cnt, uint32_t start, uint32_t size,
                                         uint32_t depth, unsigned* err) {
    const uint32_t c = seg_class(A, size);
    put_seg(A, c, atomicAdd(&cnt[c], 1u), Seg{start, size, depth, 0}, err);
}

// push_seg for a whole warp: every lane calls it (converged) and the lanes
// with `want` push their segment.  Lanes pushing to the same list share one
// atomic on its counter: a round can emit millions of short segments, and one
// atomic per segment on the few list counters serialises in L2.
__device__ __forceinline__ void push_seg_warp(const LsArgs& A, uint32_t* cnt, bool want, uint32_t start, uint32_t size,
                                              uint32_t depth, unsigned* err) {
    if (__ballot_sync(SSS_FULL, want) == 0) return;
    const uint32_t cls = want ? seg_class(A, size) : (uint32_t)LC_COUNT;
    const unsigned peers = __match_any_sync(SSS_FULL, cls);
    if (!want) return;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t leader = (uint32_t)__ffs(peers) - 1u;
    const uint32_t rank = (uint32_t)__popc(peers & ((1u << lane) - 1u));
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(&cnt[cls], (uint32_t)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    put_seg(A, cls, base + rank, Seg{start, size, depth, 0}, err);
}

// Dynamic work distribution: the next unit for the whole CTA (units vary a lot
// in cost, so a static block-to-unit map leaves a long tail).  A CTA's first
// unit is its own index, the counter hands out the ones past the grid: a grid
// larger than its work ends without touching the counter (10^4 atomics on one
// address take 9 us).
__device__ __forceinline__ uint32_t cta_next_unit(uint32_t* counter) {
    __shared__ uint32_t s_unit;
    __syncthreads();
    if (threadIdx.x == 0) s_unit = gridDim.x + atomicAdd(counter, 1u);
    __syncthreads();
    return s_unit;
}

// Candidates for the reference member of a group of `cnt` strings starting at
// `start` with depth `depth`: fixed pseudo-random members, the t-th from
// ref_pick(.., t) (results do not depend on the choice).  The finishers and
// the large path take the longest of several candidates: a member's LCP with
// the reference is capped by the reference's length, so a short reference keeps
// every longer member that shares its whole remainder in one group.  Always
// taking the first member would let an input whose order follows the strings'
// lengths or shared prefixes peel off a few strings per round.
__device__ __forceinline__ uint32_t ref_mix(uint32_t start, uint32_t cnt, uint32_t depth, uint32_t t) {
    uint32_t x = start * 0x9E3779B9u ^ (depth + 0x7F4A7C15u) * 0x85EBCA6Bu ^ cnt * 0xC2B2AE35u ^ t * 0x27D4EB2Fu;
    x ^= x >> 16;
    x *= 0x7FEB352Du;
    x ^= x >> 15;
    x *= 0x846CA68Bu;
    x ^= x >> 16;
    return x;
}
__device__ __forceinline__ uint32_t ref_pick(uint32_t start, uint32_t cnt, uint32_t depth, uint32_t t = 0) {
    return cnt > 1 ? ref_mix(start, cnt, depth, t) % cnt : 0u;
}

// Start of a sort: the call's arguments into the context's device state,
// identity order and LCP 0 over positions q0 .. q1 (or both as they are, with
// A.keep), no LCPs to recompute, and
// the given initial segments (`table`, in device memory, goes through
// k_ls_classify instead) on their lists.  One launch in place of an upload per
// list, two memsets and the identity kernel.
constexpr uint32_t LS_INLINE = 64;  // initial segments passed by value
struct LsInit {
    Seg seg[LS_INLINE];
    uint32_t n;
};
constexpr uint32_t BG_T = 256, BG_PER = 4;

__global__ void __launch_bounds__(BG_T) k_ls_begin(LsDev* __restrict__ S, const __grid_constant__ LsArgs A,
                                                   const __grid_constant__ LsInit init,
                                                   unsigned* err) {
    const uint32_t q0 = A.q0, q1 = A.q1;
    const uint32_t base = blockIdx.x * BG_T * BG_PER + threadIdx.x;
#pragma unroll
    for (uint32_t k = 0; k < BG_PER; ++k) {
        const uint32_t i = base + k * BG_T;
        if (i < q1 - q0 && !A.keep) {
            A.perm[q0 + i] = q0 + i;
            A.lcp[q0 + i] = 0;
        }
    }
    // the words holding the bits of q0 .. q1 - 1 (at most one word per 32
    // positions and one more: every block clears its share)
    const uint32_t w0 = q0 >> 5, nw = ((q1 - 1) >> 5) - w0 + 1;
    for (uint32_t w = blockIdx.x * BG_T + threadIdx.x; w < nw; w += gridDim.x * BG_T) A.fixmap[w0 + w] = 0;
    if (blockIdx.x != 0) return;
    if (threadIdx.x < 8) S->cnt[threadIdx.x] = S->work[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        S->args = A;
        S->rounds = 0;
    }
    __syncthreads();
    if (threadIdx.x < init.n) {
        const Seg s = init.seg[threadIdx.x];
        push_seg(A, S->cnt, s.start, s.size, s.depth, err);
    }
}

// every segment of >= 2 strings of a device table onto its list
__global__ void __launch_bounds__(BG_T) k_ls_classify(LsDev* __restrict__ S, const Seg* __restrict__ table, uint32_t m,
                                                      unsigned* err) {
    for (uint32_t k0 = blockIdx.x * BG_T; k0 < m; k0 += gridDim.x * BG_T) {
        const uint32_t k = k0 + threadIdx.x;
        const Seg s = k < m ? table[k] : Seg{0, 0, 0, 0};
        push_seg_warp(S->args, S->cnt, s.size >= 2, s.start, s.size, s.depth, err);
    }
}

// ---------------------------------------------------------------------------
// CTA finisher: completely sorts one segment of <= CAP strings.  Most strings
// are decided by the first iteration, whose one group is sorted by buckets and
// ranks (a call on 1,000 strings: 29 us with the merge sort of (group, key, index),
// which was 18 of the kernel's 36 thousand cycles, and a kernel to prepare it;
// 15.4 us so); the merge sort orders the groups that are left.
// fresh: the positions hold the identity order, which is not read, and the first
// one's LCP is set to 0.
template <int THREADS, int CAP>
__device__ __forceinline__ void finish_segment(const Seg sg, const uint8_t* __restrict__ chars,
                                               const uint64_t* __restrict__ offs, const uint32_t* __restrict__ lens,
                                               uint32_t* __restrict__ perm, uint32_t* __restrict__ lcp, bool fresh,
                                               unsigned* err) {
    constexpr int ITEMS = CAP / THREADS;
    constexpr bool BUCKETS = THREADS >= 128;  // (two buckets per key, 16 bits each, fit the scan buffer)
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t* sHi = reinterpret_cast<uint64_t*>(smem);  // sort keys (group:16 | word>>16)
    uint64_t* sLo = sHi + CAP;                           // (word<<48 | string index)
    uint32_t* sV = reinterpret_cast<uint32_t*>(sLo + CAP);  // string index at local position
    uint32_t* sG = sV + CAP;                             // group start of element, DONE when final
    uint32_t* sGD = sG + CAP;                            // depth of group (at its start)
    uint32_t* sGM = sGD + CAP;                           // member count (at group start)
    uint32_t* sGF = sGM + CAP;                           // key format of the group (at its start)
    uint32_t* sA = sGF + CAP;                            // scan buffer
    uint32_t* sC = sA + CAP;                             // compacted active positions
    __shared__ uint32_t sh_warp[32];
    constexpr uint32_t FIN_NREF = 68;  // 64 reference words plus a 4-word block of slack
    __shared__ uint64_t refw[FIN_NREF];

    const uint32_t m = sg.size;
    const int tid = threadIdx.x;
    for (uint32_t i = tid; i < m; i += THREADS) {
        sV[i] = fresh ? sg.start + i : perm[sg.start + i];
        sG[i] = 0;
        sC[i] = i;
    }
    if (tid == 0) {
        sGD[0] = sg.depth;
        sGM[0] = m;
        if (fresh) lcp[sg.start] = 0;
    }
    __syncthreads();

    // every iteration splits a group or finishes it, so a segment of m strings
    // needs at most about 2m iterations; the bound only guards against bugs
    for (uint32_t iter = 0;; ++iter) {
        if (iter > 4u * (uint32_t)CAP + 64u) {
            if (tid == 0) atomicOr(err, ERRBIT_OVERFLOW);
            break;
        }
        // 1. compact the positions of unfinished elements
        uint32_t nact = m;
        if (iter > 0) {
            for (uint32_t i = tid; i < (uint32_t)CAP; i += THREADS) sA[i] = (i < m && sG[i] != DONE) ? 1u : 0u;
            __syncthreads();
            nact = block_exclusive_sum_inplace<THREADS, ITEMS>(sA, CAP, sh_warp);
            for (uint32_t i = tid; i < m; i += THREADS)
                if (sG[i] != DONE) sC[sA[i]] = i;
            __syncthreads();
        }

        // 2a. every group's reference: its longest member among up to
        //     REF_CAND candidates (all members of a smaller group, scanned from
        //     a pseudo-random one on, else pseudo-random ones; the earliest
        //     candidate on ties), kept at the group start in the scan buffer,
        //     which is free until step 5
        for (uint32_t j = tid; j < nact; j += THREADS) {
            const uint32_t pos = sC[j];
            if (sG[pos] != pos) continue;
            constexpr uint32_t REF_CAND = 8;
            const uint32_t c = sGM[pos], d = sGD[pos];
            uint32_t best = pos, blen = 0;
            if (c <= REF_CAND) {
                const uint32_t t0 = ref_pick(pos, c, d);
                for (uint32_t t = 0; t < c; ++t) {
                    const uint32_t q = pos + (t0 + t < c ? t0 + t : t0 + t - c);
                    const uint32_t l = lens[sV[q]];
                    if (t == 0 || l > blen) { blen = l; best = q; }
                }
            } else {
#pragma unroll
                for (uint32_t t = 0; t < REF_CAND; ++t) {
                    const uint32_t q = pos + ref_pick(pos, c, d, t);
                    const uint32_t l = lens[sV[q]];
                    if (t == 0 || l > blen) { blen = l; best = q; }
                }
            }
            sA[pos] = best;
        }
        __syncthreads();
        // the first iteration has one group, the whole segment: its reference's
        // first 512 characters from the depth on go to shared memory, so that
        // every member reads only its own string (with 16-byte loads)
        if (iter == 0) {
            const uint32_t r0 = sV[sA[0]], rl0 = lens[r0];
            for (uint32_t i = tid; i < FIN_NREF; i += THREADS) refw[i] = load_word_be(chars + offs[r0], rl0, sGD[0] + 8 * i);
            __syncthreads();
        }

        // 2b. reference-split key of every member against its group's
        //     reference; pack (group, key, index)
        for (uint32_t j = tid; j < nact; j += THREADS) {
            uint32_t pos = sC[j];
            uint32_t g = sG[pos];
            uint32_t d = sGD[g];
            const uint32_t refpos = sA[g];
            uint32_t e = sV[pos], r = sV[refpos];
            const uint8_t* rs = chars + offs[r];
            uint32_t rl = lens[r];
            uint64_t w;
            uint32_t v;
            const uint32_t f = key_fmt(rl, d);
            if (pos == g) sGF[g] = f;
            if (pos == refpos) {
                v = rl > d ? rl - d : 0u;
                v = v < VCAP ? v : VCAP;
                w = load_word_be(rs, rl, d + v);
            } else {
                const uint32_t le = lens[e];
                const uint32_t mlen = le < rl ? le : rl;
                v = (iter == 0 && mlen <= d + 8 * (FIN_NREF - 4)) ? lcp_full_w_ref(chars + offs[e], le, rl, refw, d, &w)
                                                                  : lcp_full_w(chars + offs[e], le, rs, rl, d, &w);
            }
            const uint32_t rho = (iter == 0 && (v >> 3) < FIN_NREF)
                                     ? (uint32_t)(refw[v >> 3] >> (56 - 8 * (v & 7))) & 0xFFu
                                     : (uint32_t)(load_word_be(rs, rl, d + v) >> 56);
            uint64_t k = ref_key(v, w, rho, f);
            if (BUCKETS && iter == 0) {
                sHi[j] = k;  // one group: the key alone (its index is at sV[j])
            } else {
                sHi[j] = ((uint64_t)g << 48) | (k >> 16);
                sLo[j] = (k << 48) | (uint64_t)e;
            }
        }
        __syncthreads();

        // 3. sort (group, key, index)
        bool sorted = false;
        if constexpr (BUCKETS) {
            if (iter == 0) {
                uint16_t* sP = reinterpret_cast<uint16_t*>(sG);  // (one group: all zero, set again below)
                sorted = block_bucket_sort<THREADS, ITEMS, 2 * CAP>(sHi, sV, reinterpret_cast<uint16_t*>(sA), sLo, sP,
                                                                    m, sGF[0]);
                uint64_t k[ITEMS];
                uint32_t e[ITEMS];
#pragma unroll
                for (int t = 0; t < ITEMS; ++t) {
                    const uint32_t j = tid + t * THREADS;
                    if (j >= m) continue;
                    const uint32_t slot = sorted ? sP[j] : j;
                    k[t] = sHi[slot];
                    e[t] = sV[slot];
                }
                __syncthreads();
#pragma unroll
                for (int t = 0; t < ITEMS; ++t) {
                    const uint32_t j = tid + t * THREADS;
                    if (j >= m) continue;
                    sHi[j] = k[t] >> 16;
                    sLo[j] = (k[t] << 48) | (uint64_t)e[t];
                    sG[j] = 0;
                }
                __syncthreads();
            }
        }
        if (!sorted) block_merge_sort128_fit<THREADS, ITEMS>(sHi, sLo, nact);

        // 5. write back, find new group boundaries, LCP at new boundaries
        for (uint32_t j = tid; j < nact; j += THREADS) {
            uint32_t pos = sC[j];
            uint64_t hi = sHi[j], lo = sLo[j];
            uint32_t g = (uint32_t)(hi >> 48);
            uint64_t k = (hi << 16) | (lo >> 48);
            sV[pos] = (uint32_t)lo;
            bool bnd = true;
            if (j > 0) {
                uint64_t hp = sHi[j - 1], lp = sLo[j - 1];
                uint32_t gp = (uint32_t)(hp >> 48);
                uint64_t kp = (hp << 16) | (lp >> 48);
                if (gp == g) {
                    bnd = (kp != k);
                    if (bnd) lcp[sg.start + pos] = sGD[g] + key_lcp(kp, k, sGF[g]);
                }
            }
            sA[j] = bnd ? pos : 0u;
        }
        __syncthreads();
        block_inclusive_max_inplace<THREADS, ITEMS>(sA, nact, sh_warp);

        // 6. member count of every new group
        for (uint32_t j = tid; j < nact; j += THREADS)
            if (sA[j] == sC[j]) sGM[sC[j]] = 0;
        __syncthreads();
        for (uint32_t j = tid; j < nact; j += THREADS) atomicAdd(&sGM[sA[j]], 1u);
        __syncthreads();

        // 7. classify: single strings and runs of equal strings are final
        uint32_t dnew[ITEMS], fnew[ITEMS];
#pragma unroll
        for (int t = 0; t < ITEMS; ++t) {
            uint32_t j = tid + t * THREADS;
            if (j < nact) {
                dnew[t] = sGD[(uint32_t)(sHi[j] >> 48)];
                fnew[t] = sGF[(uint32_t)(sHi[j] >> 48)];
            }
        }
        __syncthreads();
        bool left = false;
#pragma unroll
        for (int t = 0; t < ITEMS; ++t) {
            uint32_t j = tid + t * THREADS;
            if (j >= nact) continue;
            uint32_t pos = sC[j];
            uint32_t ng = sA[j];
            uint64_t k = (sHi[j] << 16) | (sLo[j] >> 48);
            uint32_t cnt = sGM[ng];
            if (cnt == 1) {
                sG[pos] = DONE;
            } else if (key_ended(k, fnew[t])) {
                sG[pos] = DONE;
                if (pos != ng) lcp[sg.start + pos] = lens[(uint32_t)sLo[j]];
            } else {
                left = true;
                sG[pos] = ng;
                if (pos == ng) sGD[ng] = dnew[t] + key_v(k, fnew[t]) + fmt_chars(fnew[t]);
            }
        }
        if (!__syncthreads_or(left)) break;
    }
    for (uint32_t i = tid; i < m; i += THREADS) perm[sg.start + i] = sV[i];
}

// Where a finisher's segments and strings are: list `cls` of the context's
// device state (S), or explicit arrays (S == NULL), or the one segment of a call
// whose positions are fresh (segs NULL too).
struct FinIn {
    const LsDev* S;
    uint32_t cls;
    GPtr<const Seg> segs;
    uint32_t count;
    GPtr<uint32_t> work;
    GPtr<const uint8_t> chars;
    GPtr<const uint64_t> offs;
    GPtr<const uint32_t> lens;
    GPtr<uint32_t> perm;
    GPtr<uint32_t> lcp;
    Seg one;
};

// the same with the state's pointers filled in; count = 0 if a list overran
__device__ __forceinline__ FinIn fin_resolve(FinIn f, unsigned* err) {
    if (f.S) {
        const LsArgs& A = f.S->args;
        f.segs.p = A.list[f.cls];
        f.count = f.S->cnt[f.cls];
        f.work.p = const_cast<uint32_t*>(&f.S->work[f.cls]);
        f.chars.p = A.chars;
        f.offs.p = A.offs;
        f.lens.p = A.lens;
        f.perm.p = A.perm;
        f.lcp.p = A.lcp;
        // the short classes share an array of cap[] entries
        const uint32_t used = f.cls <= LC_WARP ? f.S->cnt[LC_QUAD] + f.S->cnt[LC_WARP] : f.count;
        if (used > A.cap[f.cls] || f.count > A.cap[f.cls]) {
            if (threadIdx.x == 0) atomicOr(err, ERRBIT_OVERFLOW);
            f.count = 0;
        }
    }
    return f;
}

// Segments, one CTA at a time.
template <int THREADS, int CAP>
__device__ __forceinline__ void finish_list(const FinIn& in, unsigned* err) {
    __shared__ FinIn f;  // in shared memory: its pointers would cost the loop 10 registers
    if (threadIdx.x == 0) f = fin_resolve(in, err);
    __syncthreads();
    const uint32_t nseg = f.count;
    for (uint32_t i = blockIdx.x; i < nseg; i = f.segs.p ? cta_next_unit(f.work) : nseg)
        finish_segment<THREADS, CAP>(f.segs.p ? f.segs[i] : f.one, f.chars, f.offs, f.lens, f.perm, f.lcp, !f.segs.p,
                                     err);
}

template <int THREADS, int CAP>
__global__ void __launch_bounds__(THREADS) k_finish(const FinIn in, unsigned* err) {
    finish_list<THREADS, CAP>(in, err);
}

// k_finish held to two CTAs per SM (the 512-thread class)
template <int THREADS, int CAP>
__global__ void __launch_bounds__(THREADS, 2) k_finish2(const FinIn in, unsigned* err) {
    finish_list<THREADS, CAP>(in, err);
}

// Group finisher: W consecutive lanes of a warp (W = 32, or QUAD_W for the
// shortest segments, 32 / W segments per warp) completely sort one segment of
// <= W strings, lane i of the group holding position i.  Same rounds as the CTA
// finisher (reference-split key of every unfinished member against its group's
// reference, sort by (group, key, index), split), with the sort a bitonic
// network in registers.  Every lane of the warp runs every round (the loop
// ends when no lane of the warp is left unfinished); a group whose segment is
// finished, or that has none (`has` false), carries its lanes along unchanged.
__device__ __forceinline__ void warp_cas128(uint64_t& hi, uint64_t& lo, uint32_t gl, uint32_t j, bool up) {
    uint64_t ohi = __shfl_xor_sync(SSS_FULL, hi, j), olo = __shfl_xor_sync(SSS_FULL, lo, j);
    bool keep_min = (((gl & j) == 0) == up);
    bool other_less = key128_less(ohi, olo, hi, lo);
    if (keep_min ? other_less : key128_less(hi, lo, ohi, olo)) {
        hi = ohi;
        lo = olo;
    }
}

template <int W>
__device__ __forceinline__ void finish_group_segment(const Seg sg, uint32_t e, const uint8_t* __restrict__ chars,
                                                     const uint64_t* __restrict__ offs,
                                                     const uint32_t* __restrict__ lens, uint32_t* __restrict__ perm,
                                                     uint32_t* __restrict__ lcp, unsigned* err) {
    static_assert(W >= 2 && W <= 32 && (W & (W - 1)) == 0, "group width is a power of two <= 32");
    constexpr uint64_t DONE_BIT = 1ull << 47;  // in the low word, above the 32-bit index and the lane (5 bits)
    constexpr unsigned WMASK = W == 32 ? ~0u : ((1u << W) - 1u);
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t gl = lane & (W - 1);  // lane within the group
    const uint32_t gb = lane - gl;       // the group's first lane
    const uint32_t m = sg.size <= (uint32_t)W ? sg.size : (uint32_t)W;
    const bool live = gl < m;
    // bitonic span, uniform over the warp: the group width, or for a whole-warp
    // group the next power of two >= m (lanes past it hold padding and sit out)
    const uint32_t span = W < 32 ? (uint32_t)W : (m <= 2u ? 2u : (1u << (32 - __clz((int)(m - 1)))));
    uint32_t len = live ? lens[e] : 0u;
    uint64_t off = live ? offs[e] : 0ull;  // (both follow the string from lane to lane)
    uint32_t g = 0, gd = sg.depth, gc = m;  // group start (within the segment), depth, member count
    bool done = !live;
    for (uint32_t iter = 0;; ++iter) {
        if (__ballot_sync(SSS_FULL, !done) == 0) break;
        if (iter > 4u * W + 8u) {
            if (!done) atomicOr(err, ERRBIT_OVERFLOW);
            break;
        }
        // the reference of the lane's group: its longest member, ties broken by
        // a pseudo-random rank (segmented max-scan over the group's lanes; the
        // group's last lane holds the maximum)
        uint64_t best = live ? ((uint64_t)len << 32) | (ref_mix(g, gc, gd, gl + 1u) & 0xFFFFFF00u) | gl : 0ull;
        const uint32_t gs = live ? g : gl;
#pragma unroll
        for (uint32_t o = 1; o < (uint32_t)W; o <<= 1) {
            const uint64_t y = __shfl_up_sync(SSS_FULL, best, o, W);
            if (gl >= gs + o) best = y > best ? y : best;
        }
        best = __shfl_sync(SSS_FULL, best, gb + (live ? g + gc - 1u : gl));
        const uint32_t rlane = (uint32_t)best & 0xFFu;
        const uint64_t roff = __shfl_sync(SSS_FULL, off, gb + rlane);
        const uint32_t rl = __shfl_sync(SSS_FULL, len, gb + rlane);
        const uint32_t f = key_fmt(rl, gd);
        uint64_t hi, lo;
        if (!done) {
            const uint8_t* rs = chars + roff;
            uint64_t w;
            uint32_t v;
            if (gl == rlane) {
                v = rl > gd ? rl - gd : 0u;
                v = v < VCAP ? v : VCAP;
                w = load_word_be(rs, rl, gd + v);
            } else {
                v = lcp_full_w(chars + off, len, rs, rl, gd, &w);
            }
            uint64_t k = ref_key(v, w, (uint32_t)(load_word_be(rs, rl, gd + v) >> 56), f);
            hi = ((uint64_t)g << 48) | (k >> 16);
            lo = (k << 48) | (uint64_t)e << 5 | gl;
        } else if (live) {
            hi = (uint64_t)gl << 48;  // a finished string is the only member of group `gl`
            lo = DONE_BIT | (uint64_t)e << 5 | gl;
        } else {
            hi = ~0ull;
            lo = ~0ull;
        }
        for (uint32_t kk = 2; kk <= span; kk <<= 1) {
            const bool up = (gl & kk) == 0 || kk == span;
            for (uint32_t j = kk >> 1; j > 0; j >>= 1) warp_cas128(hi, lo, gl, j, up);
        }
        // lane j of the group now holds position j; groups kept their ranges
        const uint32_t gg = (uint32_t)(hi >> 48);
        const uint64_t k = (hi << 16) | (lo >> 48);
        const bool fin = !live || (lo & DONE_BIT);
        const uint32_t src = gb + ((uint32_t)lo & 31u);
        e = (uint32_t)(lo >> 5);
        len = __shfl_sync(SSS_FULL, len, src);
        off = __shfl_sync(SSS_FULL, off, src);
        if (!live) len = 0;
        const uint64_t hp = __shfl_up_sync(SSS_FULL, hi, 1, W), lp = __shfl_up_sync(SSS_FULL, lo, 1, W);
        const uint32_t gp = (uint32_t)(hp >> 48);
        const uint64_t kp = (hp << 16) | (lp >> 48);
        bool bnd = true;
        if (gl > 0 && !fin && gp == gg && !(lp & DONE_BIT)) {
            bnd = (kp != k);
            if (bnd) lcp[sg.start + gl] = gd + key_lcp(kp, k, f);
        }
        // new group start: inclusive max-scan of boundary positions
        uint32_t ng = bnd ? gl : 0u;
#pragma unroll
        for (uint32_t o = 1; o < (uint32_t)W; o <<= 1) {
            uint32_t y = __shfl_up_sync(SSS_FULL, ng, o, W);
            if (gl >= o) ng = ng > y ? ng : y;
        }
        const unsigned bm = (__ballot_sync(SSS_FULL, bnd) >> gb) & WMASK;
        const unsigned after = gl < (uint32_t)W - 1u ? (bm & (~0u << (gl + 1))) : 0u;
        const uint32_t end = after ? (uint32_t)(__ffs(after) - 1) : m;
        const uint32_t cnt = (end > ng ? end : ng + 1) - ng;
        if (!fin) {
            if (cnt == 1) {
                done = true;
            } else if (key_ended(k, f)) {
                done = true;
                if (gl != ng) lcp[sg.start + gl] = len;
            } else {
                done = false;
                g = ng;
                gc = cnt;
                gd = gd + key_v(k, f) + fmt_chars(f);
            }
        } else {
            done = true;
            g = gl;
            gc = 1;
        }
    }
    if (live) perm[sg.start + gl] = e;
}

// Short segments, 32 / W per warp: segment i is segs[i], or segs[-i] for the
// class that fills its array downwards.  A warp's first three units are fixed,
// the counter hands out the rest.  Bound by the chain of dependent loads of a unit
// (counter, segment, strings, their offsets and lengths, characters), so the first
// three of them run ahead: while a unit is sorted, the next one's strings, the
// second's segments and the third's number are on their way; a string's offset and
// length move with it between the lanes.  The batch of 4,096 instances: 323 -> 290 us
// for its segments of 2 to 4 strings, 99 -> 95 for those of up to 32.
template <int W>
__global__ void __launch_bounds__(32 * WF_WARPS, 4) k_finish_group(const FinIn in, unsigned* err) {
    constexpr uint32_t G = 32u / W;
    __shared__ FinIn f;
    if (threadIdx.x == 0) f = fin_resolve(in, err);
    __syncthreads();
    const uint32_t nseg = f.count;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t step = gridDim.x * WF_WARPS * G;
    const auto load_seg = [&](uint32_t i0) {
        const uint32_t i = i0 + lane / W;
        return i0 < nseg && i < nseg ? (f.cls == LC_WARP ? *(f.segs - i) : f.segs[i]) : Seg{0, 0, 0, 0};
    };
    const auto load_string = [&](const Seg& sg) {
        return (lane & (W - 1)) < sg.size ? f.perm[sg.start + (lane & (W - 1))] : 0u;
    };
    uint32_t i0 = (blockIdx.x * WF_WARPS + (threadIdx.x >> 5)) * G, i1 = i0 + step, i2 = i1 + step;
    Seg s0 = load_seg(i0), s1 = load_seg(i1);
    uint32_t e0 = load_string(s0);
    while (i0 < nseg) {
        uint32_t i3 = ~0u;
        if (lane == 0 && i2 < nseg) i3 = 3 * step + atomicAdd(f.work, G);
        const Seg s2 = load_seg(i2);
        const uint32_t e1 = load_string(s1);
        finish_group_segment<W>(s0, e0, f.chars, f.offs, f.lens, f.perm, f.lcp, err);
        i0 = i1;
        i1 = i2;
        i2 = __shfl_sync(SSS_FULL, i3, 0);
        s0 = s1;
        s1 = s2;
        e0 = e1;
    }
}

constexpr size_t finish_smem(int cap) { return (size_t)cap * (8 + 8 + 4 * 7); }
// sort_emit's shared memory: keys, scratch, indices, sorted order, counters.
// The scratch is one word per key (or the low words of a 128-bit merge sort); the
// counters are 16 bits wide, two per key (the next power of two).  A CTA of 512
// threads takes 4,352 strings: as many, in steps of 256, as two of them on an SM
// have memory for.
constexpr int emit_buckets(int cap) { return cap <= 2048 ? 4096 : 8192; }
constexpr int emit_merge_items(int threads, int cap) { return cap / threads >= 8 ? 8 : 4; }
constexpr size_t emit_smem(int, int cap) { return (size_t)cap * (8 + 8 + 4 + 2) + 2 * (size_t)emit_buckets(cap); }

// ---------------------------------------------------------------------------
// Large path.
// the uncached LCP scan, kept out of line: it is the rare path of k_lg_ext
// (strings that go on past the 1,024 cached reference characters)
__device__ __noinline__ uint32_t lcp_full_w_outline(const uint8_t* a, uint32_t la, const uint8_t* b, uint32_t lb,
                                                    uint32_t d, uint64_t* w) {
    return lcp_full_w(a, la, b, lb, d, w);
}

// The round's tiles, and every segment's reference (a warp each): the longest of
// REF_CAND pseudo-random members (the earliest candidate on ties).  A member's
// LCP with the reference is capped by the reference's length, so a short
// reference leaves every longer member that shares its whole remainder in one
// group, and an input whose shared prefixes grow with the length (nested copies
// of one template) then sheds only a fraction of the segment per round.
__global__ void __launch_bounds__(256) k_lg_tiles(const LsDev* __restrict__ S) {
    const LsArgs& A = S->args;
    const uint32_t nt = S->plan.ntiles, ns = S->plan.ns;
    const uint32_t gt = blockIdx.x * 256 + threadIdx.x, nthreads = gridDim.x * 256, lane = threadIdx.x & 31;
    for (uint32_t s = gt >> 5; s < ns; s += nthreads >> 5) {
        constexpr uint32_t REF_CAND = 8;
        const Seg sg = A.info[s].seg;
        uint64_t best = 0, off = 0;
        uint32_t pos = sg.start;
        if (lane < REF_CAND) {
            pos = sg.start + ref_pick(sg.start, sg.size, sg.depth, lane);
            const uint32_t e = A.perm[pos];
            best = ((uint64_t)A.lens[e] << 32) | (uint64_t)(REF_CAND - lane);
            off = A.offs[e];
        }
        uint64_t win = best;
#pragma unroll
        for (uint32_t o = REF_CAND / 2; o > 0; o >>= 1) {
            const uint64_t x = __shfl_xor_sync(SSS_FULL, win, o);
            win = x > win ? x : win;
        }
        if (lane < REF_CAND && best == win) {
            const uint32_t rl = (uint32_t)(best >> 32), f = key_fmt(rl, sg.depth);
            A.ref[s] = LgRef{{A.chars + off}, rl, f, pos, 0};
            A.segfmt[s] = f;
        }
    }
    for (uint32_t g = gt; g < nt; g += nthreads) {
        uint32_t a = 0, c = ns;
        while (a + 1 < c) {
            const uint32_t mid = (a + c) >> 1;
            if (A.tile0[mid] <= g) a = mid;
            else c = mid;
        }
        const Seg sg = A.info[a].seg;
        const uint32_t t = g - A.tile0[a], begin = sg.start + t * LG_TILE, e = sg.start + sg.size;
        A.tiles[g] = LgTile{a, begin, e - begin < (uint32_t)LG_TILE ? e : begin + LG_TILE, t};
    }
}

// Keys: every member's LCP with its segment's reference from the depth on, and
// its next characters.  What the member loop needs of the call and the tile sits
// in shared memory: in registers next to the word stream it spills at the six
// CTAs per SM this kernel lives on.  It is a chain of dependent gathers, bound by
// latency until enough are in flight, so a unit is a whole tile (four members a
// thread) only where there are two tiles or more per CTA; below that a quarter
// tile.  Strings that go on past the cached reference characters are compared
// with the reference in memory, twice the loads.  300,007 strings of 16 to 1,000
// characters: 168 us with whole tiles (293 of them on 912 CTAs) and 512 cached
// characters, 104 us with quarter tiles, 57 us with 1,024 cached characters too.
struct ExtTile {
    GPtr<const uint8_t> chars;
    GPtr<const uint64_t> offs;
    GPtr<const uint32_t> lens;
    GPtr<const uint32_t> perm;
    GPtr<uint64_t> K;
    LgRef ref;
    uint32_t depth, begin, end;
};

__global__ void __launch_bounds__(LG_T, 6) k_lg_ext(const LsDev* __restrict__ S) {
    constexpr uint32_t NREF = 132;  // 128 words (1,024 characters) plus a 4-word block of slack
    __shared__ uint64_t refw[NREF];
    __shared__ ExtTile P;
    const LsArgs& A = S->args;
    if (threadIdx.x == 0) {
        P.chars.p = A.chars;
        P.offs.p = A.offs;
        P.lens.p = A.lens;
        P.perm.p = A.perm;
        P.K.p = A.K;
    }
    const uint32_t sub = S->plan.ntiles < 2 * gridDim.x ? 2u : 0u;  // log2 of units per tile
    for (uint32_t g = blockIdx.x; g < S->plan.ntiles << sub; g += gridDim.x) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const LgTile tl = A.tiles[g >> sub];
            const uint32_t u = (uint32_t)LG_TILE >> sub, b = tl.begin + (g & ((1u << sub) - 1u)) * u;
            P.ref = A.ref[tl.s];
            P.depth = A.info[tl.s].seg.depth;
            P.begin = b;
            P.end = b + u < tl.end ? b + u : tl.end;
        }
        __syncthreads();
        const uint32_t d = P.depth;
        if (P.begin >= P.end) continue;
        if (threadIdx.x < NREF) refw[threadIdx.x] = load_word_be(P.ref.chars, P.ref.len, d + 8 * threadIdx.x);
        __syncthreads();
        for (uint32_t q = P.begin + threadIdx.x; q < P.end; q += LG_T) {
            const uint32_t rl = P.ref.len;
            uint64_t w;
            uint32_t v;
            if (q == P.ref.pos) {
                v = rl > d ? rl - d : 0u;
                v = v < VCAP ? v : VCAP;
                w = load_word_be(P.ref.chars, rl, d + v);
            } else {
                uint32_t e = P.perm[q];
                uint32_t le = P.lens[e];
                uint32_t mlen = le < rl ? le : rl;
                v = (mlen <= d + 8 * (NREF - 4)) ? lcp_full_w_ref(P.chars + P.offs[e], le, rl, refw, d, &w)
                                                 : lcp_full_w_outline(P.chars + P.offs[e], le, P.ref.chars, rl, d, &w);
            }
            uint32_t rho = (v >> 3) < NREF ? (uint32_t)(refw[v >> 3] >> (56 - 8 * (v & 7))) & 0xFFu
                                           : (uint32_t)(load_word_be(P.ref.chars, rl, d + v) >> 56);
            P.K[q] = ref_key(v, w, rho, P.ref.fmt);
        }
    }
}

// Sort positions [bs, bs+m) (m <= CAP) by (key, index) in one CTA, write the
// indices back (of the keys a bucket's first and last), set the LCP at every key change (d + key_lcp) and emit
// the groups of equal keys: runs of equal strings get lcp = length, other groups
// become segments at depth d + v + C.  The first position's LCP is left alone.
// Reads tK/tV (from_t) or K/perm fully before writing K/perm.  False (nothing
// written) if the keys need a merge sort of more than its capacity.
// Bound by the instructions and barriers of its phases (65 k cycles of a CTA of
// 4,096 strings before, 47 k now: 11 k to rank, 11 k to write back, 9 k to load
// and reduce, 7 k for the bits).  The range buckets and the 1,024 segments of
// about 4,096 strings of the 4.19M-string sort take 147 us (306 us with the
// merge sort alone), the 4,096-instance batch's 1.63 ms (2.10 ms).
template <int THREADS, int CAP>
__device__ __forceinline__ bool sort_emit(unsigned char* smem, bool from_t, uint32_t bs, uint32_t m, uint32_t d,
                                          uint32_t f, LsDev* S, unsigned* err) {
    const LsArgs& A = S->args;  // S and err are kernel parameters: no registers held through the sort
    __shared__ uint32_t s_d, s_f;
    if (threadIdx.x == 0) {
        s_d = d;
        s_f = f;
    }
    constexpr int ITEMS = (CAP + THREADS - 1) / THREADS, NB = emit_buckets(CAP);
    constexpr int MI = emit_merge_items(THREADS, CAP);
    static_assert(THREADS * MI <= CAP, "the merge sort pads its arrays to THREADS * MI");
    uint64_t* sK = reinterpret_cast<uint64_t*>(smem);
    uint64_t* sR = sK + CAP;
    uint32_t* sV = reinterpret_cast<uint32_t*>(sR + CAP);
    uint16_t* sC = reinterpret_cast<uint16_t*>(sV + CAP);
    uint16_t* sP = sC + NB;  // the sorted order: position -> slot
    {
        const uint64_t* srcK = (from_t ? A.tK : A.K) + bs;
        const uint32_t* srcV = (from_t ? A.tV : A.perm) + bs;
        uint64_t k[ITEMS];
        uint32_t v[ITEMS];
#pragma unroll
        for (int t = 0; t < ITEMS; ++t) {
            const uint32_t i = threadIdx.x + t * THREADS;
            k[t] = i < m ? srcK[i] : 0ull;
            v[t] = i < m ? srcV[i] : 0u;
        }
#pragma unroll
        for (int t = 0; t < ITEMS; ++t) {
            const uint32_t i = threadIdx.x + t * THREADS;
            if (i < m) {
                sK[i] = k[t];
                sV[i] = v[t];
            }
        }
    }
    if (!block_bucket_sort<THREADS, ITEMS, NB>(sK, sV, sC, sR, sP, m, f)) {
        if (m > (uint32_t)(THREADS * MI)) return false;
        block_merge_sort_pairs<THREADS, MI>(sK, sV, sR, m);
        for (uint32_t i = threadIdx.x; i < m; i += THREADS) sP[i] = (uint16_t)i;
        __syncthreads();
    }
    uint32_t* perm = A.perm;
    uint32_t* lcp = A.lcp;
    d = s_d;
    f = s_f;
    // Write the order back and list the groups of equal keys in shared memory
    // (start | size << 16, in the sort's scratch): pushed as they are found, each
    // step would wait for an atomic's way to L2 and back.
    uint32_t* sG = reinterpret_cast<uint32_t*>(sR);
    __shared__ uint32_t s_ng;
    if (threadIdx.x == 0) s_ng = 0;
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t i0 = 0; i0 < m; i0 += THREADS) {  // uniform trip count: whole warps shuffle
        const uint32_t i = i0 + threadIdx.x;
        if (i - lane >= m) break;
        const uint32_t slot = sP[i < m ? i : m - 1];
        const uint64_t k = sK[slot];
        // the keys next to the warp's 32: before the first, after the last
        uint64_t kx = 0;
        if (lane == 0 && i > 0) kx = sK[sP[i - 1]];
        if (lane == 31 && i + 1 < m) kx = sK[sP[i + 1]];
        uint64_t kp = __shfl_up_sync(SSS_FULL, k, 1);
        if (lane == 0) kp = kx;
        const bool bnd = i == 0 || i >= m || kp != k;  // starts a group (past the end: closes the last one)
        const unsigned bm = __ballot_sync(SSS_FULL, bnd);
        const bool goes_on = __ballot_sync(SSS_FULL, lane == 31 && i + 1 < m && kx == k) != 0;
        const bool ended = key_ended(k, f);
        uint32_t c = 0;
        if (i < m) {
            const uint32_t e = sV[slot];
            perm[bs + i] = e;
            if (bnd) {
                if (i > 0) lcp[bs + i] = d + key_lcp(kp, k, f);
                if (!ended) {
                    const unsigned after = lane < 31 ? bm >> (lane + 1) : 0u;
                    c = after ? (uint32_t)__ffs((int)after) : 32u - lane;
                    if (!after && goes_on) {
                        // past the warp: the group's end by doubling steps, then halving ones
                        uint32_t lo = i - lane + 32, step = 1;
                        while (lo + step < m && sK[sP[lo + step]] == k) {
                            lo += step;
                            step *= 2;
                        }
                        uint32_t hi = lo + step < m ? lo + step : m;  // equal at lo; at hi it is not, or hi == m
                        while (hi - lo > 1) {
                            const uint32_t mid = (lo + hi) >> 1;
                            if (sK[sP[mid]] == k) lo = mid;
                            else hi = mid;
                        }
                        c = hi - i;
                    }
                }
            } else if (ended) {
                lcp[bs + i] = A.lens[e];  // a run of equal strings
            }
            if (from_t && (i == 0 || i + 1 == m)) A.K[bs + i] = k;  // for the LCP at the bucket's ends
        }
        const unsigned gm = __ballot_sync(SSS_FULL, c >= 2);
        if (gm) {
            uint32_t base = 0;
            if (lane == 0) base = atomicAdd(&s_ng, (uint32_t)__popc(gm));
            base = __shfl_sync(SSS_FULL, base, 0);
            if (c >= 2) sG[base + (uint32_t)__popc(gm & ((1u << lane) - 1u))] = i | c << 16;
        }
    }
    __syncthreads();
    const uint32_t ng = s_ng;
    for (uint32_t j0 = threadIdx.x - lane; j0 < ng; j0 += THREADS) {  // whole warps: push_seg_warp
        const uint32_t j = j0 + lane;
        const uint32_t x = j < ng ? sG[j] : 0u, i = x & 0xFFFFu;
        uint32_t dn = 0;
        if (j < ng) dn = d + key_v(sK[sP[i]], f) + fmt_chars(f);
        push_seg_warp(A, S->cnt, j < ng, bs + i, x >> 16, dn, err);
    }
    return true;
}

// An equality bucket, or a range bucket too large for its CTA, is copied to its
// place as it is; in a run of equal strings (ended) the LCPs are the lengths.  Eight
// strings of a thread in flight.
template <int THREADS>
__device__ __forceinline__ void copy_run(const LsArgs& A, uint32_t bs, uint32_t m, bool ended, uint32_t part,
                                         uint32_t parts) {
    constexpr uint32_t PER = 8;
    for (uint64_t i0 = (uint64_t)part * THREADS * PER + threadIdx.x; i0 < m; i0 += (uint64_t)parts * THREADS * PER) {
        uint32_t v[PER], l[PER];
#pragma unroll
        for (uint32_t t = 0; t < PER; ++t) v[t] = i0 + t * THREADS < m ? A.tV[bs + i0 + t * THREADS] : 0u;
#pragma unroll
        for (uint32_t t = 0; t < PER; ++t) l[t] = ended && i0 + t * THREADS < m ? A.lens[v[t]] : 0u;
#pragma unroll
        for (uint32_t t = 0; t < PER; ++t) {
            const uint64_t i = i0 + t * THREADS;
            if (i >= m) break;
            A.perm[bs + i] = v[t];
            if (ended && i > 0) A.lcp[bs + i] = l[t];
        }
    }
}

// A bucket of more strings than this is left to all the CTAs of the round's last
// kernel, by an entry (start, size, ended) in memory that is free by then.  4.19M
// suffixes of one repeated character (rounds of one bucket each): 127 ms of copies
// by one CTA a round of 137 in all, 6.4 ms in all so.  (Each CTA reads every entry, so
// they are few.)
constexpr uint32_t BIG_RUN = 1u << 17;
static_assert(sizeof(LgRef) >= sizeof(Seg) && BIG_RUN > 2 * (uint32_t)MED_CAP, "one reference per large segment");
__device__ __forceinline__ Seg* big_runs(const LsArgs& A) { return reinterpret_cast<Seg*>(static_cast<LgRef*>(A.ref)); }

// One CTA per bucket of the partitioned segments, and per whole segment that
// fits: range buckets and whole segments are sorted in shared memory, groups of
// equal keys become new segments at depth d + v + C.  The sort is a chain of
// short phases between barriers, so two CTAs of 512 threads on an SM overlap
// where one of 1024 threads waits (k_lg_direct keeps the segments of more than
// CAP strings).
template <int THREADS, int CAP>
__global__ void __launch_bounds__(THREADS, 65536 / (64 * THREADS)) k_lg_buckets(LsDev* S, unsigned* err) {
    extern __shared__ __align__(16) unsigned char smem[];
    const LsArgs& A = S->args;
    const uint32_t nb = S->plan.pbuckets, small0 = S->plan.npart + S->plan.nbig;
    const uint32_t n = nb + S->plan.ns - small0;
    for (uint32_t g = blockIdx.x; g < n; g = cta_next_unit(&S->work[5])) {
        const bool bucket = g < nb;
        const uint32_t sidx = bucket ? warp_last_le(A.bk0, S->plan.npart, g) : small0 + (g - nb);
        const Seg sg = A.info[sidx].seg;
        const uint32_t f = A.segfmt[sidx];
        uint32_t bs = sg.start, m = sg.size, b = 0;
        if (bucket) {
            b = g - A.bk0[sidx];
            const uint32_t* bst = A.bst + (size_t)sidx * (LG_NBMAX + 1) + b;
            bs = bst[0];
            const uint32_t be = bst[1];
            if (bs < sg.start || be > sg.start + sg.size || be < bs) {
                if (threadIdx.x == 0) atomicOr(err, ERRBIT_OVERFLOW);
                continue;
            }
            m = be - bs;
            if (m == 0) continue;
        }
        const bool eq = (b & 1u) != 0;
        if (!eq && m <= (uint32_t)CAP && sort_emit<THREADS, CAP>(smem, bucket, bs, m, sg.depth, f, S, err)) continue;
        if (!bucket) {
            if (threadIdx.x == 0) A.redo[atomicAdd(&S->cnt[6], 1u)] = sidx;  // at most one entry per segment
            continue;
        }
        const uint64_t k = A.tK[bs];
        const bool ended = eq && key_ended(k, f);
        if (m <= BIG_RUN) copy_run<THREADS>(A, bs, m, ended, 0, 1);
        if (threadIdx.x != 0) continue;
        if (m > BIG_RUN) big_runs(A)[atomicAdd(&S->cnt[7], 1u)] = Seg{bs, m, ended ? 1u : 0u, 0};
        A.K[bs] = k;
        A.K[bs + m - 1] = A.tK[bs + m - 1];
        if (!eq) {
            // oversized range bucket: another round at this depth.  Its members
            // have distinct keys, so the LCPs across its two ends depend on which
            // members end up first and last: recomputed after the last round.
            const uint32_t be = bs + m;
            push_seg(A, S->cnt, bs, m, sg.depth, err);
            if (bs > sg.start) atomicOr(&A.fixmap[bs >> 5], 1u << (bs & 31u));
            if (be < sg.start + sg.size) atomicOr(&A.fixmap[be >> 5], 1u << (be & 31u));
        } else if (m >= 2 && !ended) {
            push_seg(A, S->cnt, bs, m, sg.depth + key_v(k, f) + fmt_chars(f), err);
        }
    }
}

// LCP at the first position of every non-first, non-empty bucket of segment s.
__device__ __forceinline__ void lg_seams(const LsArgs& A, uint32_t s) {
    const LgSegInfo si = A.info[s];
    const uint32_t* bst = A.bst + (size_t)s * (LG_NBMAX + 1);
    const uint32_t nbk = 2 * si.nb - 1;
    const uint32_t f = A.segfmt[s];
    for (uint32_t b = threadIdx.x; b < nbk; b += blockDim.x) {
        const uint32_t bs = bst[b], be = bst[b + 1];
        if (be > bs && bs > si.seg.start && be <= si.seg.start + si.seg.size)
            A.lcp[bs] = si.seg.depth + key_lcp(A.K[bs - 1], A.K[bs], f);
    }
}

// The last kernel of a round.  Bucket seams of the partitioned segments (their
// buckets are sorted by now) and the copies of the largest buckets, then the
// segments of more than a bucket CTA's and at most DIRECT_CAP strings, and those it
// handed on: one CTA sorts a whole segment by its keys (no sampling, classification
// or scatter).  The last CTA to end decides whether the round loop goes on: another
// round while segments were pushed, the round limit holds and no capacity error
// occurred (loop = 1: inside a captured loop).
template <int THREADS, int CAP>
__global__ void __launch_bounds__(THREADS) k_lg_direct(LsDev* S, unsigned* err, cudaGraphConditionalHandle h,
                                                       int loop) {
    extern __shared__ __align__(16) unsigned char smem[];
    const LsArgs& A = S->args;
    const uint32_t nbig = S->plan.nbig, npart = S->plan.npart;
    for (uint32_t s = blockIdx.x; s < npart; s += gridDim.x) lg_seams(A, s);
    const uint32_t nruns = S->cnt[7];
    for (uint32_t i = 0; i < nruns; ++i) {
        const Seg run = big_runs(A)[i];
        copy_run<THREADS>(A, run.start, run.size, run.depth != 0, blockIdx.x, gridDim.x);
    }
    const uint32_t n = nbig + S->cnt[6];
    for (uint32_t i = blockIdx.x; i < n; i = cta_next_unit(&S->work[6])) {
        const uint32_t sidx = i < nbig ? npart + i : A.redo[i - nbig];
        const LgSegInfo si = A.info[sidx];
        if (si.seg.size > (uint32_t)CAP) continue;
        sort_emit<THREADS, CAP>(smem, false, si.seg.start, si.seg.size, si.seg.depth, A.segfmt[sidx], S, err);
    }
    if (!loop) return;
    __syncthreads();
    if (threadIdx.x != 0) return;
    __threadfence();
    if (atomicAdd(&S->work[7], 1u) + 1u != gridDim.x) return;
    const uint32_t r = ++S->rounds;
    bool more = atomicAdd(&S->cnt[LC_LARGE], 0u) > 0;
    if (more && r >= A.limit) {
        atomicOr(err, ERRBIT_OVERFLOW);
        more = false;
    }
    if (*(volatile unsigned*)err & ERRBIT_OVERFLOW) more = false;
    cudaGraphSetConditional(h, more ? 1u : 0u);
}

// LCP with the predecessor at the positions marked by k_lg_buckets, from the
// final order (full comparison; there are at most two per oversized bucket).
// One bit per position: a scan of n / 8 bytes.  The first position sorted keeps
// its 0.
__global__ void __launch_bounds__(256) k_fix_seams(const LsDev* __restrict__ S) {
    const LsArgs& A = S->args;
    const uint32_t q0 = A.q0, q1 = A.q1;
    for (uint32_t w = (q0 >> 5) + blockIdx.x * 256 + threadIdx.x; w <= (q1 - 1) >> 5; w += gridDim.x * 256) {
        for (uint32_t m = A.fixmap[w]; m; m &= m - 1) {
            const uint32_t q = 32 * w + (uint32_t)__ffs(m) - 1;
            if (q <= q0 || q >= q1) continue;
            const uint32_t a = A.perm[q - 1], b = A.perm[q];
            const uint32_t la = A.lens[a], lb = A.lens[b], n = la < lb ? la : lb;
            WordStream sa, sb;
            sa.init(A.chars + A.offs[a], la, 0);
            sb.init(A.chars + A.offs[b], lb, 0);
            uint32_t r = n;
            for (uint32_t k = 0; k < n; k += 8) {
                const uint64_t x = sa.next() ^ sb.next();
                if (x) {
                    const uint32_t c = k + ((uint32_t)__clzll((long long)x) >> 3);
                    r = c < n ? c : n;
                    break;
                }
            }
            A.lcp[q] = r;
        }
    }
}

__global__ void k_dist(const uint32_t* __restrict__ lens, uint32_t n, const uint32_t* __restrict__ perm,
                       const uint32_t* __restrict__ lcp, uint32_t* __restrict__ dist) {
    uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    uint32_t left = r > 0 ? lcp[r] : 0;
    uint32_t right = r + 1 < n ? lcp[r + 1] : 0;
    uint32_t m = left > right ? left : right;
    uint32_t i = perm[r];
    uint64_t d = (uint64_t)m + 1;
    dist[i] = d < lens[i] ? (uint32_t)d : lens[i];
}

__global__ void k_check_input(const uint8_t* __restrict__ chars, uint64_t n_chars, const uint64_t* __restrict__ offs,
                              const uint32_t* __restrict__ lens, uint32_t n, unsigned* err) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t o = offs[i];
    uint32_t l = lens[i];
    if (o > n_chars || (uint64_t)l > n_chars - o || l >= 0x80000000u) {
        atomicOr(err, ERRBIT_CHECK);
        return;
    }
    for (uint32_t k = 0; k < l; ++k)
        if (chars[o + k] == 0) {
            atomicOr(err, ERRBIT_CHECK);
            return;
        }
}

// The size-class knobs of the local sort; 0 takes the default (values are clamped
// by the API already).  Two defaults are rules:
//  * cta_cap: a call whose segments all fit the CTA finisher (<= 2,048 strings)
//    runs no rounds, which cost it 28 us more (1,000 strings: 27 us against 55).
//    With larger segments the rounds run anyway, and the bucket CTAs sort a
//    segment of more than 256 strings faster than the finisher, whose every
//    iteration sorts (group, key, index): 11 serving requests 397 us with 2,048,
//    337 with 256; the 4,096-instance batch 4839 and 4804.
//  * direct_cap: 8,192, but k_lg_plan may have the segments above direct_min, a
//    bucket CTA's capacity, partitioned.  A given value holds as it is.
struct LsKnobs {
    uint32_t warp_cap, cta_cap, direct_cap, bucket_target, direct_min;
};
static LsKnobs ls_knobs(const sss_params& prm, bool rounds) {
    LsKnobs k;
    k.warp_cap = prm.warp_cap ? std::min(prm.warp_cap, 32u) : 32u;
    k.cta_cap = prm.cta_cap ? std::min(std::max(prm.cta_cap, (uint32_t)TINY_CAP), (uint32_t)MED_CAP)
                            : (rounds ? 256u : (uint32_t)MED_CAP);
    k.direct_cap = prm.direct_cap ? std::min(std::max(prm.direct_cap, k.cta_cap), (uint32_t)DIRECT_CAP)
                                  : (uint32_t)DIRECT_CAP;
    k.direct_min = prm.direct_cap ? k.direct_cap : (uint32_t)BK_CAP;
    k.bucket_target = prm.bucket_target ? std::min(std::max(prm.bucket_target, 256u), 4096u) : 2048u;
    return k;
}

// bucket CTA: the small one when its capacity is twice the target or more
bool small_buckets(uint32_t target) { return target <= (uint32_t)BKS_CAP / 2; }

// Work memory of the local sort: fills the pointers and capacities of a.
void carve_ls(Arena& ar, uint32_t n, uint32_t p, const sss_params& prm, LsArgs& a) {
    const LsKnobs kn = ls_knobs(prm, true);  // the one with more large segments
    a.cap[LC_QUAD] = a.cap[LC_WARP] = n / 2 + 2;
    a.cap[LC_TINY] = n / (kn.warp_cap + 1) + 2;
    a.cap[LC_SMALL] = n / (TINY_CAP + 1) + 2;
    a.cap[LC_MED] = n / (SM_CAP + 1) + 2;
    a.cap[LC_LARGE] = n / (kn.cta_cap + 1) + p + 2;  // every large segment holds > cta_cap strings
    a.K = ar.take<uint64_t>(n);
    a.tK = ar.take<uint64_t>(n);
    a.tV = ar.take<uint32_t>(n);
    a.list[LC_QUAD] = ar.take<Seg>(a.cap[LC_QUAD]);
    a.list[LC_WARP] = a.list[LC_QUAD] ? a.list[LC_QUAD] + (a.cap[LC_WARP] - 1) : nullptr;
    for (uint32_t c = LC_TINY; c <= LC_LARGE; ++c) a.list[c] = ar.take<Seg>(a.cap[c]);
    a.segfmt = ar.take<uint32_t>(a.cap[LC_LARGE]);
    a.fixmap = ar.take<uint32_t>(n / 32 + 1);
    carve_sp(ar, n, a.cap[LC_LARGE], n / (kn.direct_min + 1) + p + 2, a);
    a.warp_max = kn.warp_cap;
    a.med_max = kn.cta_cap;
    a.direct_max = kn.direct_cap;
    a.direct_min = kn.direct_min;
    a.target = kn.bucket_target;
    a.bucket_cap = small_buckets(kn.bucket_target) ? BKS_CAP : BK_CAP;
    a.limit = 100000u;
}

// Grid sizes follow the number of strings in four steps: a launch of more CTAs
// than there is work costs up to 3 us for a grid that only finds nothing to do.
// s is the share of the full grid: 1/8 up to 2^17 strings, then 1/4, 1/2, 1.
struct LsGrid {
    uint32_t sm, div;
    uint32_t of(uint32_t per_sm) const { return std::max(1u, sm * per_sm / div); }
};
uint32_t ls_grid_class(uint32_t nr) { return nr <= (1u << 17) ? 0u : nr <= (1u << 18) ? 1u : nr <= (1u << 19) ? 2u : 3u; }
LsGrid ls_grid(sss_ctx* ctx, uint32_t cls) { return LsGrid{(uint32_t)std::max(1, ctx->sm_count), 8u >> cls}; }

// One finisher: grid CTAs over `in`.
sss_status launch_finisher(sss_ctx* ctx, uint32_t cls, uint32_t grid, const FinIn& in) {
    switch (cls) {
        case LC_QUAD:
            return sss_launch(ctx, "ls_finish_quad", k_finish_group<QUAD_W>, dim3(grid), dim3(32 * WF_WARPS), 0, in, ctx->d_err);
        case LC_WARP:
            return sss_launch(ctx, "ls_finish_warp", k_finish_group<32>, dim3(grid), dim3(32 * WF_WARPS), 0, in, ctx->d_err);
        case LC_TINY:
            return sss_launch(ctx, "ls_finish_tiny", k_finish<TINY_T, TINY_CAP>, dim3(grid), dim3(TINY_T),
                              finish_smem(TINY_CAP), in, ctx->d_err);
        case LC_SMALL:
            return sss_launch(ctx, "ls_finish_small", k_finish<SM_T, SM_CAP>, dim3(grid), dim3(SM_T),
                              finish_smem(SM_CAP), in, ctx->d_err);
        default:
            return sss_launch(ctx, "ls_finish_cta", k_finish2<MED_T, MED_CAP>, dim3(grid), dim3(MED_T),
                              finish_smem(MED_CAP), in, ctx->d_err);
    }
}

FinIn list_input(sss_ctx* ctx, uint32_t cls) {
    FinIn f{};
    f.S = static_cast<const LsDev*>(ctx->d_ls);
    f.cls = cls;
    return f;
}

// CTAs of a finisher after a round loop (the counts are on the device)
uint32_t finisher_grid(const LsGrid& g, uint32_t cls) {
    static const uint32_t per_sm[5] = {8, 8, 16, 8, 2};
    return g.of(per_sm[cls]);
}

}  // namespace

size_t need_local_sort(uint32_t n, uint32_t p, const sss_params& prm) {
    Arena ar;
    LsArgs a{};
    carve_ls(ar, n, p, prm, a);
    return ar.off + 256;
}

static bool g_attr_done[64];

static sss_status set_ls_attributes(sss_ctx* ctx) {
    if (!g_attr_done[ctx->device & 63]) {
        SSS_CUDA(cudaFuncSetAttribute(k_finish2<MED_T, MED_CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)finish_smem(MED_CAP)));
        SSS_CUDA(cudaFuncSetAttribute(k_finish<TINY_T, TINY_CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)finish_smem(TINY_CAP)));
        SSS_CUDA(cudaFuncSetAttribute(k_finish<SM_T, SM_CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)finish_smem(SM_CAP)));
        SSS_CUDA(cudaFuncSetAttribute(k_lg_buckets<BK_T, BK_CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)emit_smem(BK_T, BK_CAP)));
        SSS_CUDA(cudaFuncSetAttribute(k_lg_buckets<BKS_T, BKS_CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)emit_smem(BKS_T, BKS_CAP)));
        SSS_CUDA(cudaFuncSetAttribute(k_lg_direct<DIRECT_T, DIRECT_CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)emit_smem(DIRECT_T, DIRECT_CAP)));
        g_attr_done[ctx->device & 63] = true;
    }
    return SSS_OK;
}

sss_status impl_local_sort(sss_ctx* ctx, Arena& ar, const StrIn& in, uint32_t p, const sss_params& prm,
                           uint32_t* perm, uint32_t* lcp) {
    std::vector<Seg> init;
    for (uint32_t i = 0; i < p; ++i) {
        uint32_t lo = part_lo(in.n, p, i), hi = part_lo(in.n, p, i + 1);
        init.push_back(Seg{lo, hi - lo, 0, 0});
    }
    return impl_sort_segments(ctx, ar, in, init, prm, perm, lcp);
}

// One round of the multi-CTA path, planned on the device from the segments the
// previous round pushed: keys, partition of the large segments, bucket sorts,
// seams and whole-segment sorts.  Segments up to cta_cap strings stay on their
// lists: they are finished once, after the last round (one launch per class
// over all rounds' segments in place of one per round).
static sss_status launch_round(sss_ctx* ctx, const LsGrid& g, bool small, cudaGraphConditionalHandle h,
                               int loop) {
    LsDev* S = static_cast<LsDev*>(ctx->d_ls);
    const LsDev* cS = S;
    SSS_TRY(sss_launch(ctx, "ls_lg_plan", k_lg_plan, dim3(1), dim3(1024), 0, S, ctx->d_err));
    SSS_TRY(sss_launch(ctx, "ls_lg_tiles", k_lg_tiles, dim3(g.of(4)), dim3(256), 0, cS));
    SSS_TRY(sss_launch(ctx, "ls_lg_ext", k_lg_ext, dim3(g.div == 8 ? 3 * g.sm : 6 * g.sm), dim3(LG_T), 0, cS));
    SSS_TRY(sss_launch(ctx, "ls_lg_samples", k_lg_samples, dim3(std::max(g.sm, g.of(4))), dim3(SP_T), 0, cS));
    SSS_TRY(sss_launch(ctx, "ls_lg_classify", k_lg_classify, dim3(g.of(6)), dim3(LG_T), 0, cS));
    SSS_TRY(sss_launch(ctx, "ls_lg_offsets", k_lg_rowscan, dim3(g.of(4)), dim3(256), 0, cS));
    SSS_TRY(sss_launch(ctx, "ls_lg_scatter", k_lg_scatter, dim3(g.of(8)), dim3(LG_T), 0, cS, ctx->d_err));
    if (small)
        SSS_TRY(sss_launch(ctx, "ls_lg_buckets", k_lg_buckets<BKS_T, BKS_CAP>, dim3(std::max(g.sm, g.of(4))),
                           dim3(BKS_T), emit_smem(BKS_T, BKS_CAP), S, ctx->d_err));
    else
        SSS_TRY(sss_launch(ctx, "ls_lg_buckets", k_lg_buckets<BK_T, BK_CAP>, dim3(std::max(g.sm, g.of(2))),
                           dim3(BK_T), emit_smem(BK_T, BK_CAP), S, ctx->d_err));
    return sss_launch(ctx, "ls_lg_direct", k_lg_direct<DIRECT_T, DIRECT_CAP>, dim3(g.sm), dim3(DIRECT_T),
                      emit_smem(DIRECT_T, DIRECT_CAP), S, ctx->d_err, h, loop);
}

// The rounds, the finishers and the seam fix as one graph: a while node whose
// body is one round, the finishers as parallel branches after it, then the
// seams.  Its kernels take the context's device state only, so one graph per
// grid class and bucket CTA (eight at most, kept in the context) serves every
// call; captured per call address, a sort of new inputs paid for a capture.
static sss_status sort_graph(sss_ctx* ctx, uint32_t gcls, bool small, cudaGraphExec_t* out) {
    sss_ctx::LsGraph& slot = ctx->ls_graphs[2 * gcls + (small ? 1 : 0)];
    if (slot.exec) {
        *out = slot.exec;
        return SSS_OK;
    }
    for (cudaStream_t* s : {&ctx->cap_stream, &ctx->cap_stream2, &ctx->cap_stream3})
        if (!*s) SSS_CUDA(cudaStreamCreateWithFlags(s, cudaStreamNonBlocking));
    for (cudaEvent_t& e : ctx->cap_event)
        if (!e) SSS_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    const LsGrid g = ls_grid(ctx, gcls);
    cudaGraph_t graph;
    SSS_CUDA(cudaGraphCreate(&graph, 0));
    cudaStream_t saved = ctx->stream;
    ctx->capturing = true;
    sss_status st = SSS_OK;
    cudaGraphConditionalHandle h;
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node = nullptr;
    cudaError_t ce = cudaGraphConditionalHandleCreate(&h, graph, 1, cudaGraphCondAssignDefault);
    cp.conditional.handle = h;
    if (ce == cudaSuccess) ce = cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &cp);
    // the body: one round
    if (ce == cudaSuccess) {
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        ce = cudaStreamBeginCaptureToGraph(ctx->cap_stream, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
        if (ce == cudaSuccess) {
            ctx->stream = ctx->cap_stream;
            st = launch_round(ctx, g, small, h, 1);
            const cudaError_t ee = cudaStreamEndCapture(ctx->cap_stream, &body);
            if (ce == cudaSuccess) ce = ee;
        }
    }
    // after it: the finishers side by side, then the seams
    if (st == SSS_OK && ce == cudaSuccess) {
        ce = cudaStreamBeginCaptureToGraph(ctx->cap_stream, graph, &node, nullptr, 1, cudaStreamCaptureModeThreadLocal);
        if (ce == cudaSuccess) {
            cudaStream_t br[3] = {ctx->cap_stream, ctx->cap_stream2, ctx->cap_stream3};
            static const uint32_t order[3][2] = {{LC_MED, LC_COUNT}, {LC_SMALL, LC_TINY}, {LC_WARP, LC_QUAD}};
            ce = cudaEventRecord(ctx->cap_event[0], br[0]);
            for (int b = 1; b < 3 && ce == cudaSuccess; ++b) ce = cudaStreamWaitEvent(br[b], ctx->cap_event[0], 0);
            for (int b = 0; b < 3 && st == SSS_OK; ++b) {
                ctx->stream = br[b];
                for (uint32_t c : order[b])
                    if (c != LC_COUNT && st == SSS_OK) st = launch_finisher(ctx, c, finisher_grid(g, c), list_input(ctx, c));
            }
            for (int b = 1; b < 3; ++b) {
                if (ce == cudaSuccess) ce = cudaEventRecord(ctx->cap_event[b], br[b]);
                if (ce == cudaSuccess) ce = cudaStreamWaitEvent(br[0], ctx->cap_event[b], 0);
            }
            ctx->stream = br[0];
            if (st == SSS_OK)
                st = sss_launch(ctx, "ls_fix_seams", k_fix_seams, dim3(g.of(4)), dim3(256), 0,
                                static_cast<const LsDev*>(ctx->d_ls));
            const cudaError_t ee = cudaStreamEndCapture(ctx->cap_stream, &graph);
            if (ce == cudaSuccess) ce = ee;
        }
    }
    ctx->capturing = false;
    ctx->stream = saved;
    cudaGraphExec_t ex = nullptr;
    if (st == SSS_OK && ce == cudaSuccess) ce = cudaGraphInstantiate(&ex, graph, 0);
    if (st != SSS_OK || ce != cudaSuccess) {
        cudaGetLastError();
        cudaGraphDestroy(graph);
        return st != SSS_OK ? st : sss_fail(ctx, SSS_ERR_CUDA, std::string("sort graph: ") + cudaGetErrorString(ce));
    }
    slot.graph = graph;
    slot.exec = *out = ex;
    return SSS_OK;
}

sss_status impl_sort_segments(sss_ctx* ctx, Arena& ar, const StrIn& in, const std::vector<Seg>& init,
                              const sss_params& prm, uint32_t* perm, uint32_t* lcp, const Seg* d_init) {
    return impl_sort_segments_range(ctx, ar, in, init, prm, perm, lcp, 0, in.n, d_init);
}

// The call's arguments for a sort of positions [q0, q1) with work memory from ar.
static LsArgs ls_args(const sss_ctx* ctx, Arena& ar, const StrIn& in, const sss_params& prm, bool rounds,
                      uint32_t* perm, uint32_t* lcp, uint32_t q0, uint32_t q1) {
    LsArgs A{};
    carve_ls(ar, in.n, 1, prm, A);
    A.med_max = ls_knobs(prm, rounds).cta_cap;
    const uint32_t sm = (uint32_t)std::max(1, ctx->sm_count);
    A.few = 2 * sm;
    A.few_alone = sm / 8;
    A.chars = in.chars;
    A.offs = in.offs;
    A.lens = in.lens;
    A.perm = perm;
    A.lcp = lcp;
    A.q0 = q0;
    A.q1 = q1;
    return A;
}

// Sort the segments on the lists (`have` of each class): the rounds while there
// are large ones, the finishers, the seams.
static sss_status run_sort(sss_ctx* ctx, const LsArgs& A, const sss_params& prm, const uint32_t (&have)[LC_COUNT]) {
    LsDev* S = static_cast<LsDev*>(ctx->d_ls);
    if (have[LC_LARGE] == 0) {
        // nothing for the rounds: the finishers over the initial segments
        const uint32_t sm = (uint32_t)std::max(1, ctx->sm_count);
        const uint32_t qpb = WF_WARPS * (32 / QUAD_W);
        const uint32_t grid[5] = {std::min((have[LC_QUAD] + qpb - 1) / qpb, sm * 8),
                                  std::min((have[LC_WARP] + WF_WARPS - 1) / WF_WARPS, sm * 16),
                                  std::min(have[LC_TINY], sm * 32), std::min(have[LC_SMALL], sm * 16),
                                  std::min(have[LC_MED], sm * 4)};
        for (uint32_t c = LC_MED + 1; c-- > LC_QUAD;) SSS_TRY(launch_finisher(ctx, c, grid[c], list_input(ctx, c)));
        return SSS_OK;
    }
    const uint32_t gcls = ls_grid_class(A.q1 - A.q0);
    const bool small = small_buckets(A.target);
    if (!ctx->timing || (prm.flags & SSS_FLAG_GRAPH)) {
        cudaGraphExec_t ex;
        SSS_TRY(sort_graph(ctx, gcls, small, &ex));
        return sss_graph_launch(ctx, "ls_graph", ex);
    }
    // kernel timing is on: the same kernels launched one by one, with the next
    // round's segment count and the error word read back after every round
    const LsGrid g = ls_grid(ctx, gcls);
    uint32_t* h_next = reinterpret_cast<uint32_t*>(ctx->h_small);
    for (uint32_t rounds = 1;; ++rounds) {
        if (rounds > A.limit) return sss_fail(ctx, SSS_ERR_CUDA, "local sort: round limit exceeded");
        SSS_TRY(launch_round(ctx, g, small, cudaGraphConditionalHandle{}, 0));
        SSS_CUDA(cudaMemcpyAsync(h_next, &S->cnt[LC_LARGE], sizeof(uint32_t), cudaMemcpyDeviceToHost, ctx->stream));
        SSS_CUDA(cudaMemcpyAsync(h_next + 1, ctx->d_err, sizeof(uint32_t), cudaMemcpyDeviceToHost, ctx->stream));
        SSS_CUDA(cudaStreamSynchronize(ctx->stream));
        if (h_next[1] & ERRBIT_OVERFLOW) return sss_fail(ctx, SSS_ERR_CUDA, "local sort: device capacity check failed");
        if (h_next[0] == 0) break;
    }
    for (uint32_t c = LC_QUAD; c <= LC_MED; ++c)
        SSS_TRY(launch_finisher(ctx, c, finisher_grid(g, c), list_input(ctx, c)));
    return sss_launch(ctx, "ls_fix_seams", k_fix_seams, dim3(g.of(4)), dim3(256), 0, (const LsDev*)S);
}

sss_status impl_sort_segments_range(sss_ctx* ctx, Arena& ar, const StrIn& in, const std::vector<Seg>& init,
                                    const sss_params& prm, uint32_t* perm, uint32_t* lcp, uint32_t q0, uint32_t q1,
                                    const Seg* d_init) {
    const uint32_t n = in.n;
    if (n == 0 || q1 <= q0) return SSS_OK;
    const uint32_t nr = q1 - q0;
    const LsKnobs kn = ls_knobs(prm, false);
    SSS_TRY(set_ls_attributes(ctx));
    if (init.size() == 1 && init[0].start == q0 && init[0].size == nr && nr > (uint32_t)TINY_CAP &&
        nr <= kn.cta_cap && nr > kn.warp_cap)
        // one segment for one CTA: a single launch, nothing to prepare
        return launch_finisher(ctx, nr <= (uint32_t)SM_CAP ? LC_SMALL : LC_MED, 1,
                               FinIn{nullptr, LC_MED, {nullptr}, 1, {nullptr}, {in.chars}, {in.offs}, {in.lens}, {perm},
                                     {lcp}, init[0]});
    bool rounds = false;  // a segment that the CTA finisher cannot take
    for (const Seg& s : init) rounds = rounds || s.size > kn.cta_cap;
    const LsArgs A = ls_args(ctx, ar, in, prm, rounds, perm, lcp, q0, q1);
    SSS_TRY(sss_fits(ctx, ar));
    LsDev* S = static_cast<LsDev*>(ctx->d_ls);

    // initial segments (partitions or instances), counted by size class
    uint32_t have[LC_COUNT] = {}, m = 0;
    LsInit li{};
    for (const Seg& s : init) {
        if (s.size < 2) continue;
        const uint32_t c = s.size <= A.warp_max    ? (s.size <= (uint32_t)QUAD_W ? LC_QUAD : LC_WARP)
                           : s.size <= (uint32_t)TINY_CAP ? LC_TINY
                           : s.size <= A.med_max   ? (s.size <= (uint32_t)SM_CAP ? LC_SMALL : LC_MED)
                                                   : LC_LARGE;
        ++have[c];
        if (m < LS_INLINE) li.seg[m] = s;
        ++m;
    }
    li.n = m <= LS_INLINE ? m : 0u;
    SSS_TRY(sss_launch(ctx, "ls_init", k_ls_begin, dim3((nr + BG_T * BG_PER - 1) / (BG_T * BG_PER)), dim3(BG_T), 0, S,
                       A, li, ctx->d_err));
    if (m > LS_INLINE && d_init) {
        // more than fit in the launch's arguments, and in device memory already
        const uint32_t all = (uint32_t)init.size();
        SSS_TRY(sss_launch(ctx, "ls_classify", k_ls_classify,
                           dim3(std::min((all + BG_T - 1) / BG_T, (uint32_t)ctx->sm_count)), dim3(BG_T), 0, S, d_init,
                           all, ctx->d_err));
    } else if (m > LS_INLINE) {
        // through the second key array, free until the first scatter (every one
        // holds >= 2 strings of 8 bytes there)
        void* pin;
        SSS_TRY(sss_pinned(ctx, sizeof(Seg) * (size_t)m, &pin));
        Seg* h = static_cast<Seg*>(pin);
        for (const Seg& s : init)
            if (s.size >= 2) *h++ = s;
        Seg* table = reinterpret_cast<Seg*>(A.tK.p);
        SSS_TRY(sss_upload(ctx, table, pin, sizeof(Seg) * (size_t)m));
        SSS_TRY(sss_launch(ctx, "ls_classify", k_ls_classify,
                           dim3(std::min((m + BG_T - 1) / BG_T, (uint32_t)ctx->sm_count)), dim3(BG_T), 0, S,
                           (const Seg*)table, m, ctx->d_err));
    }
    return run_sort(ctx, A, prm, have);
}


// Refining a sorted order: groups of positions (their strings in index order)
// that are sorted by other strings, in place.  group_start[g], g < *d_groups, is
// the first position of group g, the next one's start its end (n for the last).
// impl_groups_begin puts the groups of two or more on the lists, whose counts
// (six words at *d_counts, in device memory) the caller reads back and gives to
// impl_groups_sort.
//
// The counters take one atomic per list and CTA of 1,024 groups: with one per list
// and warp, hundreds of thousands of groups took 20 us of serial atomics.
__global__ void __launch_bounds__(BG_T) k_ls_groups(LsDev* __restrict__ S, const uint32_t* __restrict__ group_start,
                                                    const uint32_t* __restrict__ d_groups, unsigned* err) {
    constexpr uint32_t PER = 4;
    __shared__ uint32_t s_cnt[LC_COUNT], s_base[LC_COUNT];
    const LsArgs& A = S->args;
    const uint32_t m = *d_groups, n = A.q1, lane = threadIdx.x & 31;
    for (uint64_t k0 = (uint64_t)blockIdx.x * BG_T * PER; k0 < m; k0 += (uint64_t)gridDim.x * BG_T * PER) {
        uint32_t start[PER], size[PER], cls[PER], place[PER];
#pragma unroll
        for (uint32_t t = 0; t < PER; ++t) {
            const uint64_t k = k0 + t * BG_T + threadIdx.x;
            start[t] = k < m ? group_start[k] : 0u;
            size[t] = k + 1 < m ? group_start[k + 1] : k < m ? n : 0u;
        }
        __syncthreads();
        if (threadIdx.x < LC_COUNT) s_cnt[threadIdx.x] = 0;
        __syncthreads();
#pragma unroll
        for (uint32_t t = 0; t < PER; ++t) {
            size[t] -= start[t];
            cls[t] = size[t] >= 2 ? seg_class(A, size[t]) : (uint32_t)LC_COUNT;
            const unsigned peers = __match_any_sync(SSS_FULL, cls[t]);
            const int leader = __ffs((int)peers) - 1;
            uint32_t base = 0;
            if ((int)lane == leader && cls[t] < LC_COUNT) base = atomicAdd(&s_cnt[cls[t]], (uint32_t)__popc(peers));
            place[t] = __shfl_sync(SSS_FULL, base, leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
        }
        __syncthreads();
        if (threadIdx.x < LC_COUNT) {
            const uint32_t c = s_cnt[threadIdx.x];
            s_base[threadIdx.x] = c ? atomicAdd(&S->cnt[threadIdx.x], c) : 0u;
        }
        __syncthreads();
#pragma unroll
        for (uint32_t t = 0; t < PER; ++t)
            if (cls[t] < LC_COUNT) put_seg(A, cls[t], s_base[cls[t]] + place[t], Seg{start[t], size[t], 0, 0}, err);
    }
}

sss_status impl_groups_begin(sss_ctx* ctx, Arena ar, const StrIn& in, const sss_params& prm, uint32_t* perm,
                             uint32_t* lcp, const uint32_t* group_start, const uint32_t* d_groups,
                             const uint32_t** d_counts) {
    LsArgs A = ls_args(ctx, ar, in, prm, false, perm, lcp, 0, in.n);
    SSS_TRY(sss_fits(ctx, ar));
    A.keep = 1;
    SSS_TRY(set_ls_attributes(ctx));
    LsDev* S = static_cast<LsDev*>(ctx->d_ls);
    const uint32_t sm = (uint32_t)std::max(1, ctx->sm_count);
    SSS_TRY(sss_launch(ctx, "ls_init", k_ls_begin, dim3(std::min((in.n + 8191) / 8192, sm * 4)), dim3(BG_T), 0, S, A,
                       LsInit{}, ctx->d_err));
    SSS_TRY(sss_launch(ctx, "ls_classify", k_ls_groups, dim3(std::min((in.n + 4 * BG_T - 1) / (4 * BG_T), sm * 8)), dim3(BG_T),
                       0, S, group_start, d_groups, ctx->d_err));
    *d_counts = S->cnt;
    return SSS_OK;
}

sss_status impl_groups_sort(sss_ctx* ctx, Arena ar, const StrIn& in, const sss_params& prm, uint32_t* perm,
                            uint32_t* lcp, const uint32_t* counts) {
    const LsArgs A = ls_args(ctx, ar, in, prm, false, perm, lcp, 0, in.n);  // as in the device state
    uint32_t have[LC_COUNT];
    std::copy(counts, counts + LC_COUNT, have);
    return run_sort(ctx, A, prm, have);
}

size_t ls_dev_bytes() { return sizeof(LsDev); }

sss_status impl_finish_segments(sss_ctx* ctx, const Seg* tiny, uint32_t ntiny, const Seg* med, uint32_t nmed,
                                const StrIn& in, uint32_t* perm, uint32_t* lcp) {
    SSS_TRY(set_ls_attributes(ctx));
    const uint32_t sm = (uint32_t)std::max(1, ctx->sm_count);
    uint32_t* work = reinterpret_cast<uint32_t*>(ctx->d_err) + 2;  // two spare words of the context
    SSS_CUDA(cudaMemsetAsync(work, 0, sizeof(uint32_t) * 2, ctx->stream));
    FinIn f{nullptr, LC_TINY, {tiny}, ntiny, {work}, {in.chars}, {in.offs}, {in.lens}, {perm}, {lcp}, {}};
    SSS_TRY(launch_finisher(ctx, LC_TINY, std::min(ntiny, sm * 32), f));
    f.cls = LC_MED;
    f.segs = med;
    f.count = nmed;
    f.work = work + 1;
    return launch_finisher(ctx, LC_MED, std::min(nmed, sm * 4), f);
}

// Smallest offset and largest end of every partition's strings: blocks of
// 4096 positions over the whole grid, each block reducing within one partition
// and folding its result into out[2i] (min) and out[2i+1] (max) with atomics
// (out pre-set by k_part_extents_init).
__global__ void k_part_extents_init(uint32_t p, unsigned long long* __restrict__ out) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < p; i += gridDim.x * blockDim.x) {
        out[2 * i] = ~0ull;
        out[2 * i + 1] = 0ull;
    }
}

__global__ void __launch_bounds__(256) k_part_extents(const uint64_t* __restrict__ offs,
                                                      const uint32_t* __restrict__ lens, uint32_t n, uint32_t p,
                                                      unsigned long long* __restrict__ out) {
    constexpr uint32_t SPAN = 4096;
    __shared__ unsigned long long s_lo[8], s_hi[8];
    for (uint64_t c = blockIdx.x; c * SPAN < n; c += gridDim.x) {
        const uint32_t a = (uint32_t)(c * SPAN);
        const uint32_t b = (uint32_t)min((uint64_t)n, (uint64_t)a + SPAN);
        // partitions are contiguous: handle the part of [a, b) in each partition it touches
        uint32_t i = (uint32_t)(((uint64_t)a * p) / n);
        while (i + 1 < p && part_lo(n, p, i + 1) <= a) ++i;
        for (uint32_t q0 = a; q0 < b; ++i) {
            const uint32_t q1 = min(b, part_lo(n, p, i + 1));
            unsigned long long lo = ~0ull, hi = 0ull;
            for (uint32_t q = q0 + threadIdx.x; q < q1; q += 256) {
                const unsigned long long o = offs[q];
                lo = o < lo ? o : lo;
                const unsigned long long e = o + lens[q];
                hi = e > hi ? e : hi;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long ol = __shfl_xor_sync(SSS_FULL, lo, o), oh = __shfl_xor_sync(SSS_FULL, hi, o);
                lo = ol < lo ? ol : lo;
                hi = oh > hi ? oh : hi;
            }
            if ((threadIdx.x & 31) == 0) {
                s_lo[threadIdx.x >> 5] = lo;
                s_hi[threadIdx.x >> 5] = hi;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int w = 1; w < 8; ++w) {
                    lo = s_lo[w] < lo ? s_lo[w] : lo;
                    hi = s_hi[w] > hi ? s_hi[w] : hi;
                }
                if (q1 > q0) {
                    atomicMin(&out[2 * i], lo);
                    atomicMax(&out[2 * i + 1], hi);
                }
            }
            __syncthreads();
            q0 = q1;
        }
    }
}

sss_status impl_part_extents(sss_ctx* ctx, const StrIn& in, uint32_t p, unsigned long long* out) {
    const uint32_t sm = (uint32_t)std::max(1, ctx->sm_count);
    SSS_TRY(sss_launch(ctx, "part_extents", k_part_extents_init, dim3((p + 255) / 256), dim3(256), 0, p, out));
    const uint32_t blocks = std::min((in.n + 4095u) / 4096u, sm * 8);
    return sss_launch(ctx, "part_extents", k_part_extents, dim3(blocks), dim3(256), 0, in.offs, in.lens, in.n, p,
                      out);
}

uint32_t finish_cap_tiny() { return TINY_CAP; }
uint32_t finish_cap_med() { return MED_CAP; }

// Suffix views of a text: string i is text[i .. i + min(n - i, max_len)).
__global__ void k_suffix_views(uint32_t n, uint32_t max_len, uint64_t* __restrict__ offs,
                               uint32_t* __restrict__ lens) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        uint32_t r = n - i;
        offs[i] = i;
        lens[i] = r < max_len ? r : max_len;
    }
}

sss_status impl_suffix_views(sss_ctx* ctx, uint32_t n, uint32_t max_len, uint64_t* offs, uint32_t* lens) {
    return sss_launch(ctx, "sfx_views", k_suffix_views, dim3(std::min((n + 255) / 256, 65535u)), dim3(256), 0, n,
                      max_len, offs, lens);
}

// Batched sorts: table positions become instance-local indices, and the
// instance's dist is (optionally) computed.  blockIdx.y splits an instance over
// several CTAs: with one each, eleven instances of 450k strings in all kept
// eleven SMs busy for 193 us.  Eight positions of a thread are in flight: 38.7M
// positions in 4,096 instances took 129 us one at a time, 58 us (5.3 TB/s) so.
__global__ void __launch_bounds__(256) k_batch_finish(const Seg* __restrict__ inst, uint32_t m,
                                                      const uint32_t* __restrict__ lens, uint32_t* __restrict__ perm,
                                                      const uint32_t* __restrict__ lcp, uint32_t* __restrict__ dist) {
    constexpr uint32_t PER = 8, SPAN = 256 * PER;
    for (uint32_t k = blockIdx.x; k < m; k += gridDim.x) {
        const Seg s = inst[k];
        for (uint64_t r0 = (uint64_t)blockIdx.y * SPAN + threadIdx.x; r0 < s.size; r0 += (uint64_t)gridDim.y * SPAN) {
            uint32_t g[PER];
#pragma unroll
            for (uint32_t t = 0; t < PER; ++t) g[t] = r0 + t * 256 < s.size ? perm[s.start + r0 + t * 256] : 0u;
#pragma unroll
            for (uint32_t t = 0; t < PER; ++t) {
                if (r0 + t * 256 >= s.size) break;
                const uint32_t r = (uint32_t)r0 + t * 256, q = s.start + r;
                if (dist) {
                    const uint32_t left = r > 0 ? lcp[q] : 0;
                    const uint32_t right = r + 1 < s.size ? lcp[q + 1] : 0;
                    const uint64_t d = (uint64_t)(left > right ? left : right) + 1;
                    dist[g[t]] = d < lens[g[t]] ? (uint32_t)d : lens[g[t]];
                }
                perm[q] = g[t] - s.start;
            }
        }
    }
}

sss_status impl_batch_finish(sss_ctx* ctx, const Seg* d_inst, uint32_t m, const uint32_t* lens, uint32_t* perm,
                             const uint32_t* lcp, uint32_t* dist) {
    // at least 64 CTAs per SM in all, so that instances of very uneven sizes even out
    const uint32_t gx = std::min<uint32_t>(m, 65535u);
    const uint32_t gy = std::max(1u, std::min(65535u, (uint32_t)ctx->sm_count * 64u / gx));
    return sss_launch(ctx, "batch_finish", k_batch_finish, dim3(gx, gy), dim3(256), 0, d_inst, m, lens, perm, lcp,
                      dist);
}

sss_status impl_dist(sss_ctx* ctx, const uint32_t* lens, uint32_t n, const uint32_t* perm, const uint32_t* lcp,
                     uint32_t* dist) {
    return sss_launch(ctx, "dist", k_dist, dim3((n + 255) / 256), dim3(256), 0, lens, n, perm, lcp, dist);
}

sss_status impl_check_input(sss_ctx* ctx, const StrIn& in) {
    return sss_launch(ctx, "check_input", k_check_input, dim3((in.n + 255) / 256), dim3(256), 0, in.chars,
                      in.n_chars, in.offs, in.lens, in.n, ctx->d_err);
}
