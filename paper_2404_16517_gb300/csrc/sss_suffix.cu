// Suffix sorting as string sorting (the extension named in Section 6,
// "Conclusion and Future Work"): the suffixes of one text are sorted as
// strings, views into the text, without copying characters.
//
// GB300 design: prefix doubling over ranks, on top of the string sort.
//  * First the suffixes truncated to H0 = 64 characters are sorted as strings
//    by the local sort (stage A); equal truncated suffixes share a rank (the
//    number of distinct smaller truncations).  On a text with short repeats
//    every rank is already distinct here, and the result is final.
//  * Otherwise the ranks of length h are doubled: the suffix at i of length
//    next = min(2h, target) is ordered by the pair (rank_h(i), rank_h(i + o)),
//    o = next - h <= h.  The second rank covers characters [o, o + h) of the
//    suffix, so the overlap [o, h) adds nothing and the pair orders the
//    suffixes on their first `next` characters, ending at the text's end
//    (a missing second rank, past the end, is the smallest).  The order by the
//    first rank is at hand, so only the groups of equal first ranks are sorted,
//    in place, by their second ranks, as 5-character strings by the same local
//    sort: every rank + 1 is written as five 7-bit digits with the top bit set
//    (no zero byte, order kept).  Equal pairs keep the suffix order (ties by
//    position).  Most suffixes of a text with some repeats are alone by then:
//    sorting all pairs anew took a 1,000,003-character text 2.21 ms in all, this
//    1.03 ms.
//  * The rounds stop when every rank is distinct or the target length
//    (max_len, else the whole text) is reached, so a text of one repeated
//    character takes log2(n / 64) rounds instead of n^2 / 2 character reads.
//  * The LCP of two adjacent suffixes adds the lengths of the rank levels on
//    which they agree, from the longest level down, then compares the fewer
//    than 64 characters that are left.
#include <algorithm>
#include <vector>

#include "sss_device.cuh"
#include "sss_internal.cuh"

namespace {

constexpr uint32_t SX_H0 = 64;    // characters of the first, direct sort
constexpr uint32_t SX_DIGITS = 5;  // characters of a rank
constexpr int SX_MAXLEV = 34;     // rank levels at most (64 .. 2^32, plus a truncated last)

// rank levels a text of n characters can need: 64, 128, ... up to the first
// length >= n, the last possibly shorter
inline uint32_t sx_levels(uint32_t n) {
    uint32_t c = 1;
    for (uint64_t h = SX_H0; h < n; h <<= 1) ++c;
    return std::min<uint32_t>(c, SX_MAXLEV);
}

struct SxLevels {
    const uint32_t* rank[SX_MAXLEV];
    uint32_t len[SX_MAXLEV];
    uint32_t count;
};

__global__ void k_sx_views(uint32_t n, uint32_t h, uint64_t* __restrict__ offs, uint32_t* __restrict__ lens) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint32_t r = n - i;
        offs[i] = i;
        lens[i] = r < h ? r : h;
    }
}

__device__ __forceinline__ void sx_put_rank(uint8_t* p, uint32_t v) {
    p[0] = (uint8_t)(0x80u | ((v >> 28) & 0x7Fu));
    p[1] = (uint8_t)(0x80u | ((v >> 21) & 0x7Fu));
    p[2] = (uint8_t)(0x80u | ((v >> 14) & 0x7Fu));
    p[3] = (uint8_t)(0x80u | ((v >> 7) & 0x7Fu));
    p[4] = (uint8_t)(0x80u | (v & 0x7Fu));
}

// views of the digit strings: string i is P[5 i .. 5 i + 5)
__global__ void k_sx_digit_views(uint32_t n, uint64_t* __restrict__ offs, uint32_t* __restrict__ lens) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        offs[i] = (uint64_t)SX_DIGITS * i;
        lens[i] = SX_DIGITS;
    }
}

// digit string of suffix i: rank_h(i + o) + 1 (0 past the end)
__global__ void k_sx_second(const uint32_t* __restrict__ rank, uint32_t n, uint32_t o, uint8_t* __restrict__ P) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        sx_put_rank(P + (size_t)SX_DIGITS * i, (uint64_t)i + o < n ? rank[i + o] + 1u : 0u);
}

// group starts of the suffixes sorted on their first h characters: position k
// starts a group unless its truncated suffix equals its predecessor's (lcp equal
// to both lengths); *dups = positions that do not
__global__ void __launch_bounds__(256) k_sx_flags(const uint32_t* __restrict__ perm, const uint32_t* __restrict__ lcp,
                                                  uint32_t n, uint32_t h, uint32_t* __restrict__ flag,
                                                  uint32_t* __restrict__ dups) {
    uint32_t d = 0;
    for (uint32_t k = blockIdx.x * 256 + threadIdx.x; k < n; k += gridDim.x * 256) {
        uint32_t f = 1;
        if (k > 0) {
            const uint32_t l = lcp[k];
            f = (l == min(n - perm[k - 1], h) && l == min(n - perm[k], h)) ? 0u : 1u;
        }
        flag[k] = f;
        d += 1u - f;
    }
    d = __reduce_add_sync(SSS_FULL, d);
    if ((threadIdx.x & 31) == 0 && d) atomicAdd(dups, d);
}

// after the groups were sorted by their digit strings: a position inside a group
// starts one of its own when its string differs from its predecessor's
__global__ void k_sx_split(const uint32_t* __restrict__ lcp, uint32_t n, uint32_t* __restrict__ flag) {
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
        if (!flag[k] && lcp[k] != SX_DIGITS) flag[k] = 1;
}

// rank of the suffix at sorted position k: the number of group starts before
// its group (exclusive sum over the starts, plus its own start, minus one); the
// groups' first positions and their number
__global__ void k_sx_ranks(const uint32_t* __restrict__ perm, const uint64_t* __restrict__ excl,
                           const uint32_t* __restrict__ flag, uint32_t n, uint32_t* __restrict__ rank,
                           uint32_t* __restrict__ group_start, uint32_t* __restrict__ groups) {
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const uint32_t f = flag[k], r = (uint32_t)(excl[k] + f - 1u);
        rank[perm[k]] = r;
        if (f) group_start[r] = k;
        if (k == n - 1) *groups = r + 1u;
    }
}

// LCP of the suffixes at sorted positions k-1 and k, truncated to max_len
__global__ void k_sx_lcp(const uint8_t* __restrict__ text, uint32_t n, uint32_t max_len,
                         const uint32_t* __restrict__ sa, SxLevels lv, uint32_t* __restrict__ lcp) {
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        if (k == 0) {
            lcp[0] = 0;
            continue;
        }
        const uint32_t i = sa[k - 1], j = sa[k];
        const uint32_t li = min(n - i, max_len), lj = min(n - j, max_len);
        const uint32_t m = li < lj ? li : lj;
        uint32_t l = 0;
        for (int t = (int)lv.count - 1; t >= 0 && l < m; --t) {
            // equal ranks at length L: equal windows of L characters (both inside the
            // text, as the suffixes differ)
            if ((uint64_t)i + l < n && (uint64_t)j + l < n && lv.rank[t][i + l] == lv.rank[t][j + l]) l += lv.len[t];
        }
        if (l < m) {
            // fewer than the shortest level's characters are left: compare them
            for (;;) {
                const uint64_t x = load_word_be(text + i, li, l), y = load_word_be(text + j, lj, l);
                if (x != y) {
                    l += word_lcp(x, y);
                    break;
                }
                l += 8;
                if (l >= m) break;
            }
        }
        lcp[k] = l < m ? l : m;
    }
}

}  // namespace

size_t need_suffix_sort(uint32_t n, const sss_params& prm) {
    Arena a;
    a.take<uint64_t>(n);                          // views
    a.take<uint32_t>(n);
    a.take<uint8_t>((size_t)SX_DIGITS * n);       // digit strings
    a.take<uint32_t>(n);                          // group flags
    a.take<uint64_t>(n);                          // their exclusive sum
    a.take<uint64_t>(n / 4096 + 4);
    a.take<uint32_t>(n);                          // group starts
    a.take<uint32_t>(4);                          // counts
    for (uint32_t t = 0; t < sx_levels(n); ++t) a.take<uint32_t>(n);  // rank levels
    a.take<char>(need_local_sort(n, 1, prm));
    return a.off + 256;
}

// Work memory: need_suffix_sort(n), with room for the rank levels of whole
// suffixes (the most rounds any max_len can take).
sss_status impl_suffix_sort(sss_ctx* ctx, char* ws, size_t ws_bytes, const uint8_t* text, uint32_t n,
                            uint32_t max_len, const sss_params& prm, uint32_t* out_sa, uint32_t* out_lcp) {
    Arena ar{ws, ws_bytes, 0};
    uint64_t* offs = ar.take<uint64_t>(n);
    uint32_t* lens = ar.take<uint32_t>(n);
    uint8_t* P = ar.take<uint8_t>((size_t)SX_DIGITS * n);
    uint32_t* flag = ar.take<uint32_t>(n);
    uint64_t* excl = ar.take<uint64_t>(n);
    uint64_t* btot = ar.take<uint64_t>(n / 4096 + 4);
    uint32_t* gstart = ar.take<uint32_t>(n);
    uint32_t* cnt = ar.take<uint32_t>(4);  // [0] equal neighbours, [1] groups
    const uint32_t nlev = sx_levels(n);
    uint32_t* lvbase[SX_MAXLEV];
    for (uint32_t t = 0; t < nlev; ++t) lvbase[t] = ar.take<uint32_t>(n);
    size_t sort_off = (ar.off + 255) & ~size_t(255);
    SSS_TRY(sss_fits(ctx, ar));
    const Arena sort_ar{ws + sort_off, ws_bytes > sort_off ? ws_bytes - sort_off : 0, 0};
    const uint32_t sm = (uint32_t)std::max(1, ctx->sm_count);
    const uint32_t grid = std::min((n + 255) / 256, sm * 16);
    const uint32_t target = max_len ? std::min(max_len, n) : n;

    // the suffixes truncated to H0 characters, sorted as strings
    uint32_t h = std::min(SX_H0, target);
    SSS_TRY(sss_launch(ctx, "sx_views", k_sx_views, dim3(grid), dim3(256), 0, n, h, offs, lens));
    {
        Arena sa = sort_ar;
        StrIn in{text, n, offs, lens, n};
        SSS_TRY(impl_local_sort(ctx, sa, in, 1, prm, out_sa, out_lcp));
    }
    if (h >= target) return SSS_OK;  // the views were the truncated suffixes themselves
    // all distinct within H0 characters: the order and the LCPs (all shorter than
    // H0, or a suffix's whole length at the text's end) are final
    SSS_CUDA(cudaMemsetAsync(cnt, 0, sizeof(uint32_t) * 4, ctx->stream));
    SSS_TRY(sss_launch(ctx, "sx_flags", k_sx_flags, dim3(grid), dim3(256), 0, (const uint32_t*)out_sa,
                       (const uint32_t*)out_lcp, n, h, flag, cnt));
    // (the pinned staging is looked up again for every use: the sorts may grow it)
    void* pin;
    SSS_TRY(sss_pinned(ctx, 64, &pin));
    uint32_t* hc = static_cast<uint32_t*>(pin);
    SSS_CUDA(cudaMemcpyAsync(hc, cnt, sizeof(uint32_t), cudaMemcpyDeviceToHost, ctx->stream));
    SSS_CUDA(cudaStreamSynchronize(ctx->stream));
    if (hc[0] == 0) return SSS_OK;
    const StrIn din{P, (uint64_t)SX_DIGITS * n, offs, lens, n};
    SSS_TRY(sss_launch(ctx, "sx_views", k_sx_digit_views, dim3(grid), dim3(256), 0, n, offs, lens));
    SxLevels lv{};
    for (;;) {
        // ranks of the order on the first h characters, and its groups on the sort's lists
        if (lv.count >= nlev) return sss_fail(ctx, SSS_ERR_CUDA, "suffix sort: too many rounds");
        uint32_t* rank = lvbase[lv.count];
        SSS_TRY(impl_scan_u32_u64(ctx, flag, n, excl, btot));
        SSS_TRY(sss_launch(ctx, "sx_ranks", k_sx_ranks, dim3(grid), dim3(256), 0, (const uint32_t*)out_sa,
                           (const uint64_t*)excl, (const uint32_t*)flag, n, rank, gstart, cnt + 1));
        lv.rank[lv.count] = rank;
        lv.len[lv.count] = h;
        ++lv.count;
        if (h >= target) break;
        const uint32_t* d_counts;
        SSS_TRY(impl_groups_begin(ctx, sort_ar, din, prm, out_sa, out_lcp, gstart, cnt + 1, &d_counts));
        SSS_TRY(sss_pinned(ctx, 64, &pin));
        hc = static_cast<uint32_t*>(pin);
        SSS_CUDA(cudaMemcpyAsync(hc, d_counts, sizeof(uint32_t) * 6, cudaMemcpyDeviceToHost, ctx->stream));
        SSS_CUDA(cudaMemcpyAsync(hc + 6, cnt + 1, sizeof(uint32_t), cudaMemcpyDeviceToHost, ctx->stream));
        SSS_CUDA(cudaStreamSynchronize(ctx->stream));
        if (hc[6] == n) break;  // every rank is distinct
        const uint32_t next = (uint32_t)std::min<uint64_t>(2ull * h, target);
        SSS_TRY(sss_launch(ctx, "sx_second", k_sx_second, dim3(grid), dim3(256), 0, (const uint32_t*)rank, n,
                           next - h, P));
        SSS_TRY(impl_groups_sort(ctx, sort_ar, din, prm, out_sa, out_lcp, hc));
        SSS_TRY(sss_launch(ctx, "sx_split", k_sx_split, dim3(grid), dim3(256), 0, (const uint32_t*)out_lcp, n, flag));
        h = next;
    }
    // out_sa holds the order (equal truncated suffixes by position); the LCPs
    return sss_launch(ctx, "sx_lcp", k_sx_lcp, dim3(grid), dim3(256), 0, text, n, target, (const uint32_t*)out_sa,
                      lv, out_lcp);
}
