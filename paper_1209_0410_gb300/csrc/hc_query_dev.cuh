// Device helpers of the query path shared by the query kernel, the exact
// brute force and the depth predictor: 16-byte row gathers, exact distances,
// the walks of a query's windows, and lower_bound on 128-bit keys.
#pragma once

#include <type_traits>

#include "hc_internal.h"
#include "hc_topk.cuh"

namespace hc {

__device__ __forceinline__ uint4 ldg16(const void* p) {
    return __ldg(reinterpret_cast<const uint4*>(p));
}

__device__ __forceinline__ uint32_t acc_vec(uint4 a, uint4 b, uint32_t acc) {
    uint32_t t;
    t = __vabsdiffu4(a.x, b.x);
    acc = __dp4a(t, t, acc);
    t = __vabsdiffu4(a.y, b.y);
    acc = __dp4a(t, t, acc);
    t = __vabsdiffu4(a.z, b.z);
    acc = __dp4a(t, t, acc);
    t = __vabsdiffu4(a.w, b.w);
    acc = __dp4a(t, t, acc);
    return acc;
}

__device__ __forceinline__ float acc_vec(uint4 a, uint4 b, float acc) {
    float t;
    t = __uint_as_float(a.x) - __uint_as_float(b.x);
    acc = fmaf(t, t, acc);
    t = __uint_as_float(a.y) - __uint_as_float(b.y);
    acc = fmaf(t, t, acc);
    t = __uint_as_float(a.z) - __uint_as_float(b.z);
    acc = fmaf(t, t, acc);
    t = __uint_as_float(a.w) - __uint_as_float(b.w);
    acc = fmaf(t, t, acc);
    return acc;
}

__device__ __forceinline__ uint32_t dist_bits(uint32_t d) { return d; }
__device__ __forceinline__ uint32_t dist_bits(float d) { return __float_as_uint(d); }

// Candidates produced per lane by one 32-row chunk: rows wider than 8 lanes
// are reduced 8 sub-batches at a time, leaving one candidate per group.
#ifndef HC_GROUP_MAX
#define HC_GROUP_MAX 8   // sub-batches (rows per lane group) loaded before reducing
#endif

template <int LPR>
struct ChunkWidth {
    static constexpr int G = LPR < HC_GROUP_MAX ? LPR : HC_GROUP_MAX;
    static constexpr int NG = LPR / G;            // groups, candidates per lane
};

// Distances of up to 32 rows (row r of the chunk has id shfl(id, r), valid for
// r < cnt) to the query.  LPR lanes read one row, 32 / LPR rows per warp
// instruction, so the chunk takes LPR sub-batches; they are processed in
// groups of G = min(LPR, 8): the G partial sums of a group are reduce-scattered
// over the LPR lanes (G - 1 shuffles, then log2(LPR / G) plain ones), after
// which lane s holds sub-batch s / (LPR / G) of the group.  out[g] is the
// packed (distance, id) candidate of that row, or kEmpty (rows past cnt, and
// the LPR / G - 1 lanes that hold a copy).
template <bool F32, int LPR>
__device__ __forceinline__ void chunk_candidates_n(const uint8_t* __restrict__ db,
                                                   uint32_t row_bytes, const uint8_t* qrow,
                                                   uint4 qv0, uint32_t id, uint32_t cnt, int lane,
                                                   uint64_t (&out)[ChunkWidth<LPR>::NG]) {
    using Acc = typename std::conditional<F32, float, uint32_t>::type;
    constexpr int RPI = 32 / LPR;
    constexpr int G = ChunkWidth<LPR>::G;
    constexpr int NG = ChunkWidth<LPR>::NG;
    constexpr int COPIES = LPR / G;
    const uint32_t s = (uint32_t)lane % LPR, g = (uint32_t)lane / LPR;
    const uint32_t vecs = row_bytes >> 4;
    const uint32_t vpl = (vecs + LPR - 1) / LPR;
#pragma unroll
    for (int gi = 0; gi < NG; ++gi) {
        Acc part[G];
#pragma unroll
        for (int j = 0; j < G; ++j) part[j] = Acc(0);
        for (uint32_t v = 0; v < vpl; ++v) {
            const uint32_t col = s + v * LPR;
            const bool colok = col < vecs;
            const uint4 qv =
                v == 0 ? qv0 : (colok ? ldg16(qrow + col * 16) : make_uint4(0, 0, 0, 0));
            uint4 rv[G];
#pragma unroll
            for (int j = 0; j < G; ++j) {
                const uint32_t r = (uint32_t)(gi * G + j) * RPI + g;
                const uint32_t rid = __shfl_sync(0xffffffffu, id, (int)r);
                rv[j] = (r < cnt && colok) ? ldg16(db + (size_t)rid * row_bytes + col * 16)
                                           : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int j = 0; j < G; ++j) part[j] = acc_vec(rv[j], qv, part[j]);
        }
        // halving steps over the top log2(G) bits of s
#pragma unroll
        for (int w = LPR / 2, half = G / 2; half >= 1; w >>= 1, half >>= 1) {
            const bool upper = (s & (uint32_t)w) != 0;
#pragma unroll
            for (int t = 0; t < half; ++t) {
                const Acc send = upper ? part[t] : part[t + half];
                const Acc keep = upper ? part[t + half] : part[t];
                part[t] = keep + __shfl_xor_sync(0xffffffffu, send, w);
            }
        }
        // plain sums over the low log2(LPR / G) bits
        Acc dsum = part[0];
#pragma unroll
        for (int w = COPIES / 2; w >= 1; w >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, w);
        const uint32_t j = s / COPIES;
        const uint32_t r = (uint32_t)(gi * G + j) * RPI + g;
        const uint32_t cid = __shfl_sync(0xffffffffu, id, (int)(r < 32 ? r : 0));
        out[gi] = (r < cnt && (s % COPIES) == 0) ? ((uint64_t)dist_bits(dsum) << 32) | cid : kEmpty;
    }
}

// Low key word of entry g (global entry index) of list L.
__device__ __forceinline__ uint64_t entry_key_lo(const IndexView& ix, uint32_t L, uint64_t g) {
    if (ix.keys_lo) return __ldg(ix.keys_lo + g);
    const uint32_t id = __ldg(ix.ids + g);
    return row_key_lo(ix.db, ix.row_bytes, ix.P, HC_IN_BOUNDS(kSiteRow, id, ix.rows) ? id : 0u,
                      L % ix.P.curves);
}

// first i in [first, first + count) (global entries of list L) with key[i] >=
// (kh, kl), else first + count; the low word is consulted only when the high
// words tie
__device__ __forceinline__ uint64_t lower_bound_range(const IndexView& ix, uint32_t L,
                                                      uint64_t first, uint32_t count,
                                                      uint64_t end, uint64_t kh, uint64_t kl) {
    while (count > 0) {
        const uint32_t step = count >> 1;
        const uint64_t mid = first + step;
        if (!HC_IN_BOUNDS(kSiteSearch, mid, end)) break;
        const uint64_t h = __ldg(ix.keys_hi + mid);
        bool less = h < kh;
        if (h == kh) less = entry_key_lo(ix, L, mid) < kl;
        if (less) {
            first = mid + 1;
            count -= step + 1;
        } else {
            count = step;
        }
    }
    return first;
}

// first i in [0, n) of list L (entries off ..) with key[i] >= (kh, kl), else n.
// With a fence (the top 48 bits of every 16th high word of the index), the
// fence words inside the list are searched first against pk = kh &
// kFenceMask: the last one below pk and the first one above it bracket the
// answer, which is then found among the at most 15 entries between them (one
// 128-byte line of high words) instead of by probes spread over the whole
// list.  Fence words equal to pk widen the bracket to the fence words that
// tie.
__device__ __forceinline__ uint32_t lower_bound_key(const IndexView& ix, uint32_t L, uint64_t off,
                                                    uint32_t n, uint64_t kh, uint64_t kl) {
    if (!ix.fence) return (uint32_t)(lower_bound_range(ix, L, off, n, off + n, kh, kl) - off);
    const uint64_t ja = (off + 15) >> kFenceShift, jb = (off + n + 15) >> kFenceShift;
    const uint64_t pk = kh & kFenceMask;
    // jl = first fence point of the list whose fence word is >= pk
    uint64_t jl = ja;
    for (uint32_t count = (uint32_t)(jb - ja); count > 0;) {
        const uint32_t step = count >> 1;
        const uint64_t mid = jl + step;
        if (!HC_IN_BOUNDS(kSiteSearch, mid, ix.fence_len)) break;
        if (__ldg(ix.fence + mid) < pk) {
            jl = mid + 1;
            count -= step + 1;
        } else {
            count = step;
        }
    }
    // entries before lo are below the key (fence point jl - 1 is); the entry
    // at hi, a fence point whose word is above pk, is not
    const uint64_t lo = jl > ja ? ((jl - 1) << kFenceShift) + 1 : off;
    uint64_t hi = off + n;
    if (jl < jb && HC_IN_BOUNDS(kSiteSearch, jl, ix.fence_len)) {
        if (__ldg(ix.fence + jl) > pk) {
            hi = jl << kFenceShift;
        } else {
            // fence points tying pk: the first one above it ends the bracket
            uint64_t ju = jl + 1;
            for (uint32_t count = (uint32_t)(jb - ju); count > 0;) {
                const uint32_t step = count >> 1;
                const uint64_t mid = ju + step;
                if (!HC_IN_BOUNDS(kSiteSearch, mid, ix.fence_len)) break;
                if (__ldg(ix.fence + mid) <= pk) {
                    ju = mid + 1;
                    count -= step + 1;
                } else {
                    count = step;
                }
            }
            if (ju < jb) hi = ju << kFenceShift;
        }
    }
    return (uint32_t)(lower_bound_range(ix, L, lo, (uint32_t)(hi - lo), off + n, kh, kl) - off);
}

// lower_bound_key of G keys (kh[g], kl[g]) in G lists (lists[g], skipped
// where on[g] is false), the G searches in lockstep so that G loads are in
// flight per lane.  Each search halves without branches (the probe picks the
// half, the length shrinks by the same amount whatever the outcome), so lanes
// searching lists of one length run the same steps: the fence points of the
// list (first word >= kh[g] & kFenceMask), the bracket, then the first entry of the
// bracket whose key is >= (kh[g], kl[g]).  pos[g] is list-relative.  Entry indexes fit 32
// bits (an index holds fewer than 2^32 entries).
template <int G>
__device__ __forceinline__ void lower_bound_lists(const IndexView& ix, const uint32_t (&lists)[G],
                                                  const bool (&on)[G], const uint64_t (&kh)[G],
                                                  const uint64_t (&kl)[G], uint32_t (&pos)[G]) {
    if (!ix.fence) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (!on[g]) continue;
            const uint64_t off = ix.list_off[lists[g]];
            pos[g] = lower_bound_key(ix, lists[g], off,
                                     (uint32_t)(ix.list_off[lists[g] + 1] - off), kh[g], kl[g]);
        }
        return;
    }
    uint64_t pk[G];
#pragma unroll
    for (int g = 0; g < G; ++g) pk[g] = kh[g] & kFenceMask;
    uint32_t off[G], end[G], base[G], len[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        off[g] = on[g] ? (uint32_t)ix.list_off[lists[g]] : 0u;
        end[g] = on[g] ? (uint32_t)ix.list_off[lists[g] + 1] : 0u;
        base[g] = (uint32_t)(((uint64_t)off[g] + 15) >> kFenceShift);   // ja
        len[g] = (uint32_t)(((uint64_t)end[g] + 15) >> kFenceShift) - base[g];
    }
    // fence points [ja, jb): the answer jl lies in [base, base + len]
    for (;;) {
        bool busy = false;
        uint64_t f[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const uint32_t mid = base[g] + (len[g] >> 1) - 1;
            const bool go = len[g] > 1 && HC_IN_BOUNDS(kSiteSearch, mid, ix.fence_len);
            f[g] = go ? __ldg(ix.fence + mid) : 0ull;
            if (!go) len[g] = min(len[g], 1u);
            busy |= go;
        }
        if (!busy) break;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (len[g] <= 1) continue;
            const uint32_t half = len[g] >> 1;
            base[g] += f[g] < pk[g] ? half : 0u;
            len[g] -= half;
        }
    }
    // jl = base (+1 when the last candidate is below pk); fence word of jl
    uint32_t jl[G];
    uint64_t fj[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const bool one = len[g] == 1 && HC_IN_BOUNDS(kSiteSearch, base[g], ix.fence_len);
        const uint64_t fb = one ? __ldg(ix.fence + base[g]) : 0ull;
        jl[g] = base[g] + (one && fb < pk[g] ? 1u : 0u);
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const uint32_t jbg = (uint32_t)(((uint64_t)end[g] + 15) >> kFenceShift);
        fj[g] = jl[g] < jbg && HC_IN_BOUNDS(kSiteSearch, jl[g], ix.fence_len)
                    ? __ldg(ix.fence + jl[g]) : ~0ull;
    }
    // brackets [base, base + len) as in lower_bound_key
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const uint32_t ja = (uint32_t)(((uint64_t)off[g] + 15) >> kFenceShift);
        const uint32_t jbg = (uint32_t)(((uint64_t)end[g] + 15) >> kFenceShift);
        const uint32_t lo = jl[g] > ja ? ((jl[g] - 1) << kFenceShift) + 1 : off[g];
        uint32_t hi = end[g];
        if (jl[g] < jbg) {
            if (fj[g] > pk[g]) {
                hi = jl[g] << kFenceShift;
            } else {
                // fence points tying pk: the first one above it ends the bracket
                uint32_t ju = jl[g] + 1;
                for (uint32_t cnt = jbg - ju; cnt > 0;) {
                    const uint32_t step = cnt >> 1;
                    const uint32_t mid = ju + step;
                    if (!HC_IN_BOUNDS(kSiteSearch, mid, ix.fence_len)) break;
                    if (__ldg(ix.fence + mid) <= pk[g]) {
                        ju = mid + 1;
                        cnt -= step + 1;
                    } else {
                        cnt = step;
                    }
                }
                if (ju < jbg) hi = ju << kFenceShift;
            }
        }
        base[g] = lo;
        len[g] = hi - lo;
    }
    // first entry of each bracket with key >= (kh, kl): the answer lies in
    // [base, base + len]
    for (;;) {
        bool busy = false;
        uint64_t h[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const uint32_t mid = base[g] + (len[g] >> 1) - 1;
            const bool go = len[g] > 1 && HC_IN_BOUNDS(kSiteSearch, mid, end[g]);
            h[g] = go ? __ldg(ix.keys_hi + mid) : 0ull;
            if (!go) len[g] = min(len[g], 1u);
            busy |= go;
        }
        if (!busy) break;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (len[g] <= 1) continue;
            const uint32_t half = len[g] >> 1;
            bool less = h[g] < kh[g];
            if (h[g] == kh[g]) less = entry_key_lo(ix, lists[g], base[g] + half - 1) < kl[g];
            base[g] += less ? half : 0u;
            len[g] -= half;
        }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
        uint32_t at = base[g];
        if (len[g] == 1 && HC_IN_BOUNDS(kSiteSearch, at, end[g])) {
            const uint64_t h = __ldg(ix.keys_hi + at);
            bool less = h < kh[g];
            if (h == kh[g]) less = entry_key_lo(ix, lists[g], at) < kl[g];
            at += less ? 1u : 0u;
        }
        if (on[g]) pos[g] = at - off[g];
    }
}

// K1 + K3 for one query: positions of the query key in lists L0, L0 + Lstep,
// ... written to pos_w[L].
__device__ __forceinline__ void query_positions(const IndexView& ix, const uint8_t* qrow,
                                                uint32_t* pos_w, int lane, uint32_t L0 = 0,
                                                uint32_t Lstep = 1) {
    const uint32_t curves = ix.P.curves;
    uint64_t khi = 0, klo = 0;
    if ((uint32_t)lane < curves) curve_key_call(qrow, ix.P, (uint32_t)lane, khi, klo);
    const uint32_t mine = (ix.lists > L0) ? (ix.lists - L0 + Lstep - 1) / Lstep : 0;
    for (uint32_t b = 0; b < mine; b += 32) {
        const uint32_t t = b + (uint32_t)lane;
        const uint32_t L = L0 + t * Lstep;
        const int c = (int)(L % curves);
        const uint64_t kh = __shfl_sync(0xffffffffu, khi, c);
        const uint64_t kl = __shfl_sync(0xffffffffu, klo, c);
        if (t < mine) {
            const uint64_t off = ix.list_off[L];
            const uint32_t n = (uint32_t)(ix.list_off[L + 1] - off);
            pos_w[L] = lower_bound_key(ix, L, off, n, kh, kl);
        }
    }
    __syncwarp();
}

// query_positions with the lanes of the warp spread over the searches: `each`
// lanes (a power of two) take one list and probe `each` points of its bracket at
// once, so a list of n entries takes log(n) / log(each + 1) rounds of one load
// instead of log2(n).  For few lists per warp.  keys: the query's key (high, low)
// on every curve.
__device__ __forceinline__ void query_positions_spread(const IndexView& ix, const ulonglong2* keys,
                                                       uint32_t* pos_w, int lane, uint32_t L0,
                                                       uint32_t Lstep) {
    const uint32_t curves = ix.P.curves;
    const uint32_t mine = ix.lists > L0 ? (ix.lists - L0 + Lstep - 1) / Lstep : 0;
    uint32_t each = 32;
    while (each > 4 && 32 / each < mine) each /= 2;
    const uint32_t i = (uint32_t)lane % each, g = (uint32_t)lane / each;
    const uint32_t group = each == 32 ? 0xFFFFFFFFu : (1u << each) - 1u;
    for (uint32_t b = 0; b < mine; b += 32 / each) {
        const uint32_t t = b + g;
        const bool on = t < mine;
        const uint32_t L = on ? L0 + t * Lstep : L0;
        const ulonglong2 key = keys[L % curves];
        const uint64_t kh = key.x, kl = key.y;
        const uint64_t off = ix.list_off[L], end = on ? ix.list_off[L + 1] : off;
        // first point in [first, first + count) where below() no longer holds
        auto search = [&](uint64_t first, uint64_t count, auto&& below) {
            while (__any_sync(0xffffffffu, count > 0)) {
                const bool last = count <= each;
                const uint64_t at = last ? i : count * (i + 1) / (each + 1);
                const bool in = at < count;
                const bool yes = in && below(first + at);
                const uint32_t n =
                    (uint32_t)__popc(__ballot_sync(0xffffffffu, yes) >> (g * each) & group);
                if (last) {
                    first += n;
                    count = 0;
                } else {
                    const uint64_t lo = n ? count * n / (each + 1) + 1 : 0;
                    const uint64_t hi = n < each ? count * (n + 1) / (each + 1) : count;
                    first += lo;
                    count = hi - lo;
                }
            }
            return first;
        };
        uint64_t lo = off, hi = end;
        if (ix.fence) {
            // as lower_bound_key: the fence words bracket the answer
            const uint64_t ja = (off + 15) >> kFenceShift, jb = (end + 15) >> kFenceShift;
            const uint64_t pk = kh & kFenceMask;
            auto word = [&](uint64_t j) {
                return HC_IN_BOUNDS(kSiteSearch, j, ix.fence_len) ? __ldg(ix.fence + j) : ~0ull;
            };
            const uint64_t jl = search(ja, jb > ja ? jb - ja : 0, [&](uint64_t j) {
                return word(j) < pk;
            });
            const bool tie = jl < jb && word(jl) == pk;
            const uint64_t ju = search(tie ? jl + 1 : jl, tie ? jb - jl - 1 : 0, [&](uint64_t j) {
                return word(j) <= pk;
            });
            if (jl > ja) lo = ((jl - 1) << kFenceShift) + 1;
            if (ju < jb) hi = ju << kFenceShift;
        }
        const uint64_t pos = search(lo, hi > lo ? hi - lo : 0, [&](uint64_t e) {
            if (!HC_IN_BOUNDS(kSiteSearch, e, end)) return false;
            const uint64_t h = __ldg(ix.keys_hi + e);
            return h < kh || (h == kh && entry_key_lo(ix, L, e) < kl);
        });
        if (on && i == 0) pos_w[L] = (uint32_t)(pos - off);
    }
    __syncwarp();
}

// The query's positions in lists L0, L0 + Lstep, ... into pos_w[L]: read
// from a batch pass when one ran (pos_in: list order, int64; pos_cm: curve-
// major uint32, entry c * partitions + j for list j * curves + c), else
// searched here.
__device__ __forceinline__ void load_positions(const IndexView& ix, const uint8_t* qrow,
                                               uint32_t* pos_w, int lane, uint32_t L0,
                                               uint32_t Lstep, const int64_t* pos_in,
                                               const uint32_t* pos_cm) {
    if (pos_cm) {
        const uint32_t curves = ix.P.curves, parts = ix.lists / curves;
        for (uint32_t L = L0 + (uint32_t)lane * Lstep; L < ix.lists; L += 32 * Lstep)
            pos_w[L] = __ldg(pos_cm + (L % curves) * parts + L / curves);
        __syncwarp();
    } else if (pos_in) {
        for (uint32_t L = L0 + (uint32_t)lane * Lstep; L < ix.lists; L += 32 * Lstep)
            pos_w[L] = (uint32_t)__ldg(pos_in + L);
        __syncwarp();
    } else {
        query_positions(ix, qrow, pos_w, lane, L0, Lstep);
    }
}

// ---------------------------------------------------------------------------
// Staged form of the window walk for rows of at most 128 bytes: the windows of
// all lists are packed back to back and walked in steps of 32 entries (a step
// may span several short windows, so short or uneven windows fill whole steps);
// the rows of the next step are copied into a per-warp shared-memory ring with
// cp.async (no registers held while they are in flight) while the current
// step's rows are reduced, a row per lane.
// Waits are the hardware's cp.async group waits.
__device__ __forceinline__ void cp_async16(uint32_t saddr, const void* g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(saddr), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The windows of the lists this warp walks (L = L0 + m Lstep), packed back
// to back: win_at[m] = first ids entry of window m (global entry index),
// win_pre[m] = number of window entries before window m.  Returns the total.
// win_at may alias pos_w (each slot is read before it is written).
__device__ __forceinline__ uint32_t pack_windows(const IndexView& ix, uint32_t depth, uint32_t L0,
                                                 uint32_t Lstep, const uint32_t* pos_w,
                                                 uint32_t* win_at, uint32_t* win_pre, int lane) {
    const uint32_t nm = ix.lists > L0 ? (ix.lists - L0 + Lstep - 1) / Lstep : 0;
    uint32_t carry = 0;
    for (uint32_t b = 0; b < nm; b += 32) {
        const uint32_t m = b + (uint32_t)lane;
        uint32_t len = 0, at = 0;
        if (m < nm) {
            const uint32_t L = L0 + m * Lstep;
            const uint64_t off = ix.list_off[L];
            const uint32_t n = (uint32_t)(ix.list_off[L + 1] - off);
            const uint32_t pos = pos_w[L];
            const uint32_t lo = pos > depth ? pos - depth : 0u;
            const uint32_t hi = (uint64_t)pos + depth < (uint64_t)n ? pos + depth : n;
            len = hi > lo && HC_IN_BOUNDS(kSiteWindow, hi, (uint64_t)n + 1) ? hi - lo : 0u;
            at = (uint32_t)(off + lo);   // index entries < 2^32
        }
        uint32_t x = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        __syncwarp();
        if (m < nm) {
            win_at[m] = at;
            win_pre[m] = carry + x - len;
        }
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
    __syncwarp();
    return carry;
}

// A lane's place in the packed windows: the window of its last entry, the
// packed entry at which that window ends, and first entry - packed entry of it.
// A lane's entries only grow, so most calls find the window they left.
struct WindowCursor {
    uint32_t m = ~0u, end = 0, base = 0;

    // id of packed entry e, or of the last one (total - 1) when e is past it; e
    // is not below the lane's last one, total > 0
    __device__ __forceinline__ uint32_t id(const IndexView& ix, const uint32_t* win_at,
                                           const uint32_t* win_pre, uint32_t nm, uint32_t total,
                                           uint32_t e) {
        e = min(e, total - 1);
        while (e >= end) {
            ++m;
            end = m + 1 < nm ? win_pre[m + 1] : total;
            base = win_at[m] - win_pre[m];
        }
        const uint32_t ent = base + e;
        if (!HC_IN_BOUNDS(kSiteEntry, ent, ix.list_off[ix.lists])) return 0u;
        const uint32_t id = __ldg(ix.ids + ent);
        return HC_IN_BOUNDS(kSiteRow, id, ix.rows) ? id : 0u;
    }

    // the window of packed entry e, so that a walk starting there need not pass
    // all before it (the largest window that starts at or before e)
    __device__ __forceinline__ void seek(const uint32_t* win_pre, uint32_t nm, uint32_t e) {
        uint32_t lo = 0, count = nm;
        while (count > 1) {
            const uint32_t half = count >> 1;
            if (win_pre[lo + half] <= e) {
                lo += half;
                count -= half;
            } else {
                count = half;
            }
        }
        m = lo - 1;
    }
};

// Rows of at most 128 bytes staged in shared memory, 32 to a stage: row r's
// 16-byte vector c lies at vector c ^ f(r) of the row, so that eight lanes
// reading vector c of eight neighbouring rows touch eight different bank groups
// (f(r) = the row's low bits, as many as the row's vector count has factors of
// two, taken from bit 3 - that many up).
struct RowSwizzle {
    uint32_t shift, mask;
    __device__ __forceinline__ explicit RowSwizzle(uint32_t vecs) {
        const uint32_t g = vecs & (0u - vecs);   // a power of two, at most 8
        mask = g - 1;
        shift = 3u - (uint32_t)(31 - __clz(g));
    }
    __device__ __forceinline__ uint32_t at(uint32_t r, uint32_t c) const {
        return c ^ ((r >> shift) & mask);
    }
};

// The two-stage pipeline of staged rows: while the copies of one step are in
// flight the step before it is reduced, a whole row per lane, so no partial sums
// cross lanes.  FULL: rows of exactly 16 LPR bytes (128 or 64).  add() takes the
// next step's ids (lane l: row l; the rows of lanes at or past cnt are copied but
// not offered), finish() reduces the last one.  ring: two stages of 32 rows,
// 128-byte aligned.  START: the first step's candidates are sorted into the list
// instead of inserted one by one (a call in the loop: with 80 registers its spills
// cost more than the insertions for k > 32 and rows over 64 bytes; elsewhere it
// gains 3-4% over all depths, 64-byte rows at k = 100 8%).
constexpr uint32_t kRingRows = 64;     // two stages of 32 rows
constexpr uint32_t kWideRing = 8192;   // bytes: two stages of walk_wide

template <bool F32, int LPR, int KR, bool FULL, bool START>
struct StagedSteps {
    const uint8_t* db;               // (values: a reference would put them in local memory)
    uint32_t row_bytes;
    uint8_t* ring;
    // the query's vectors (zero past the row) in registers, or, where they and the
    // list (or the general row layout) do not fit beside each other, read again for
    // every step (80 registers, 60,000 queries, k = 100, p = 16: 128-byte rows 1.68
    // against 1.73 ms with the vectors held; 96-byte rows at p = 200 4.6 against 5.2;
    // 64-byte rows and k = 37 are faster with them held)
    static constexpr bool kHold = FULL && (START || KR <= 2 || LPR < 8);
    const uint8_t* qrow;
    uint4 q[kHold ? 8 : 1];
    uint32_t id = 0, cnt = 0;        // of the step in flight (cnt = 0: none)
    uint32_t at = 0;                 // byte offset of its stage
    RowSwizzle sw;
    uint64_t thr;                    // the k-th candidate so far
    bool fresh;                      // no candidate so far

    __device__ __forceinline__ StagedSteps(const IndexView& ix, const uint8_t* query,
                                           uint8_t* ring_mem, const WarpTopK<KR>& top, uint32_t k)
        : db(static_cast<const uint8_t*>(ix.db)),
          row_bytes(ix.row_bytes),
          ring(ring_mem),
          qrow(query),
          sw(ix.row_bytes >> 4),
          thr(top.kth(k)) {
        fresh = START && __all_sync(0xffffffffu, top.v[0] == kEmpty);
        if constexpr (kHold)
#pragma unroll
            for (int c = 0; c < 8; ++c)
                q[c] = c < LPR && (FULL || (uint32_t)c < (row_bytes >> 4))
                           ? ldg16(qrow + c * 16)
                           : make_uint4(0, 0, 0, 0);
    }

    __device__ __forceinline__ uint4 query_vec(int c) const {
        if constexpr (kHold) return q[c];
        else return ldg16(qrow + c * 16);
    }

    __device__ __forceinline__ uint32_t other_stage() const {
        return (FULL ? 512u * LPR : 32u * row_bytes) - at;
    }

    // copies of one step: lane (c = lane % LPR, g = lane / LPR) moves vector c of
    // rows g, g + 32 / LPR, ... (vectors past the row are skipped)
    __device__ __forceinline__ void issue(uint32_t nid, uint32_t stage, int lane) {
        constexpr uint32_t RPI = 32 / LPR;
        const uint32_t c = (uint32_t)lane % LPR, g = (uint32_t)lane / LPR;
        const uint8_t* col = db + c * 16;
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(ring) + stage;
        if constexpr (FULL) {
            // 8 vectors: rows g + 4 t swap by g or g + 4; 4 vectors: rows g + 8 t by g / 2
            const uint32_t x = LPR == 8 ? c ^ g : c ^ ((g >> 1) & 3u);
            const uint32_t even = base + g * (16 * LPR) + x * 16;
            const uint32_t odd = LPR == 8 ? even ^ 64u : even;
#pragma unroll
            for (int t = 0; t < LPR; ++t) {
                const uint32_t rid = __shfl_sync(0xffffffffu, nid, (int)(g + RPI * (uint32_t)t));
                cp_async16((t & 1 ? odd : even) + 512u * (uint32_t)t,
                           col + (uint64_t)rid * (16u * LPR));
            }
        } else {
            const bool colok = c < (row_bytes >> 4);
#pragma unroll
            for (int t = 0; t < LPR; ++t) {
                const uint32_t r = g + RPI * (uint32_t)t;
                const uint32_t rid = __shfl_sync(0xffffffffu, nid, (int)r);
                if (colok)
                    cp_async16(base + r * row_bytes + sw.at(r, c) * 16,
                               col + (size_t)rid * row_bytes);
            }
        }
    }

    // Distance of the staged row `lane` to the query.  float32: a sum per
    // vector, then the vectors' sums by halves of LPR (v and v + LPR / 2, then
    // LPR / 4, ...), the order in which rows read by LPR lanes are reduced.
    __device__ __forceinline__ uint32_t distance(int lane) const {
        const uint32_t vecs = FULL ? (uint32_t)LPR : row_bytes >> 4;
        const uint8_t* row = ring + at + (uint32_t)lane * (FULL ? 16u * LPR : row_bytes);
        const uint32_t x = (LPR == 8 && FULL) ? (uint32_t)lane & 7u
                           : FULL             ? ((uint32_t)lane >> 1) & 3u
                                              : sw.at((uint32_t)lane, 0);
        auto vec = [&](int c) {
            return *reinterpret_cast<const uint4*>(row + (((uint32_t)c ^ x) << 4));
        };
        if constexpr (F32) {
            float part[LPR];
#pragma unroll
            for (int c = 0; c < LPR; ++c)
                part[c] = (uint32_t)c < vecs ? acc_vec(vec(c), query_vec(c), 0.f) : 0.f;
#pragma unroll
            for (int w = LPR / 2; w >= 1; w >>= 1)
#pragma unroll
                for (int c = 0; c < w; ++c) part[c] = part[c] + part[c + w];
            return __float_as_uint(part[0]);
        } else {
            uint32_t acc[2] = {0, 0};
#pragma unroll
            for (int c = 0; c < LPR; ++c)
                if ((uint32_t)c < vecs) acc[c & 1] = acc_vec(vec(c), query_vec(c), acc[c & 1]);
            return acc[0] + acc[1];
        }
    }

    __device__ __forceinline__ void reduce(WarpTopK<KR>& top, uint32_t k, int lane) {
        __syncwarp();   // every lane's copies have landed
        const uint32_t d = distance(lane);
        const bool live = (uint32_t)lane < cnt;
        if (START && fresh) {
            fresh = false;
            if (top.start(live ? ((uint64_t)d << 32) | id : kEmpty, lane)) {
                thr = top.kth(k);
                return;
            }
        }
        top.offer_row(d, id, live, k, thr, lane);
    }

    // between: called while the copies of both steps are in flight
    template <typename Between>
    __device__ __forceinline__ void add(uint32_t nid, uint32_t ncnt, WarpTopK<KR>& top, uint32_t k,
                                        int lane, Between&& between) {
        __syncwarp();   // every lane is done with the stage before it is refilled
        issue(nid, other_stage(), lane);
        cp_async_commit();
        between();
        if (cnt) {
            cp_async_wait<1>();
            reduce(top, k, lane);
        }
        id = nid;
        cnt = ncnt;
        at = other_stage();
    }
    __device__ __forceinline__ void finish(WarpTopK<KR>& top, uint32_t k, int lane) {
        cp_async_wait<0>();
        if (cnt) reduce(top, k, lane);
        cnt = 0;
    }
};

// The walk of a query's packed windows (rows of at most 128 bytes): steps
// part, part + parts, ... of 32 entries, the ids of the next two on their way: asked
// for before the next step's rows or (LATE) behind them.
template <bool F32, int LPR, int KR, bool FULL, bool SPLIT, bool START, bool LATE>
__device__ __forceinline__ void walk_staged(const IndexView& ix, const uint8_t* qrow, uint32_t k,
                                            const uint32_t* win_at, const uint32_t* win_pre,
                                            uint32_t nm, uint32_t total, uint32_t my_part,
                                            uint32_t my_parts, uint8_t* ring, WarpTopK<KR>& top,
                                            int lane) {
    const uint32_t part = SPLIT ? my_part : 0u, parts = SPLIT ? my_parts : 1u;
    const uint32_t steps = total / 32 + (total % 32 != 0);
    if (part >= steps) return;
    StagedSteps<F32, LPR, KR, FULL, START> pipe(ix, qrow, ring, top, k);
    WindowCursor cur;
    const uint32_t stride = 32 * parts;
    uint32_t e = 32 * part + (uint32_t)lane;
    if (part) cur.seek(win_pre, nm, e);
    auto id_of = [&](uint32_t step, uint32_t at) {
        return step < steps ? cur.id(ix, win_at, win_pre, nm, total, at) : 0u;
    };
    uint32_t id0 = id_of(part, e), id1 = id_of(part + parts, e + stride);
    for (uint32_t s = part; s < steps; s += parts) {
        uint32_t id2 = 0;
        if constexpr (!LATE) id2 = id_of(s + 2 * parts, e + 2 * stride);
        pipe.add(id0, min(32u, total - 32 * s), top, k, lane, [&] {
            if constexpr (LATE) id2 = id_of(s + 2 * parts, e + 2 * stride);
        });
        e += stride;
        id0 = id1;
        id1 = id2;
    }
    pipe.finish(top, k, lane);
}

// The same for wider rows, LPR lanes to a row: window by window in steps of 32
// entries, the next step's ids on their way.  A step's rows are read in units of
// eight 16-byte vectors per lane (vector s + v LPR of eight sub-batches of 32 /
// LPR rows), each unit copied into one of two 4 KB stages while the unit before
// it is added up; a lane reads back only what it copied itself.  A unit's sums
// are those of chunk_candidates_n, reduced in the same order.  Of every `parts`
// steps in a row this warp takes one.
template <bool F32, int LPR, int KR, bool SPLIT>
__device__ __forceinline__ void walk_wide(const IndexView& ix, const uint8_t* qrow, uint32_t k,
                                          const uint32_t* win_at, const uint32_t* win_pre,
                                          uint32_t nm, uint32_t total, uint32_t my_part,
                                          uint32_t my_parts, uint8_t* ring, WarpTopK<KR>& top,
                                          int lane) {
    using Acc = typename std::conditional<F32, float, uint32_t>::type;
    constexpr uint32_t RPI = 32 / LPR;
    constexpr int G = 8, NG = LPR / G, COPIES = LPR / G;
    const uint32_t stride = SPLIT ? 32 * my_parts : 32u;
    const uint32_t s = (uint32_t)lane % LPR, g = (uint32_t)lane / LPR;
    const uint32_t row_bytes = ix.row_bytes, vecs = row_bytes >> 4;
    const uint32_t vpl = (vecs + LPR - 1) / LPR;
    const uint8_t* db = static_cast<const uint8_t*>(ix.db);
    const uint4 qv0 = s < vecs ? ldg16(qrow + s * 16) : make_uint4(0, 0, 0, 0);
    const uint32_t slot = (uint32_t)__cvta_generic_to_shared(ring) + (uint32_t)lane * 16;

    // steps: entries base .. of the window that ends at hi; m: the window after it
    uint32_t m = 0, base = 0, hi = 0, skip = SPLIT ? my_part : 0u;
    auto next_step = [&](uint32_t& id, uint32_t& cnt) {   // cnt = 0: no more
        if (hi - base > stride) {
            base += stride;
        } else {
            base = hi;
            while (base == hi && m < nm) {
                base = win_at[m];
                const uint32_t len = (m + 1 < nm ? win_pre[m + 1] : total) - win_pre[m];
                hi = base + len;
                ++m;
                if (SPLIT) {
                    const uint32_t steps = len / 32 + (len % 32 != 0);
                    if (skip >= steps) {
                        skip -= steps;
                        base = hi;
                    } else {
                        base += 32 * skip;
                        skip += my_parts * ((steps - skip + my_parts - 1) / my_parts) - steps;
                    }
                }
            }
        }
        cnt = min(32u, hi - base);
        id = 0;
        if ((uint32_t)lane < cnt &&
            HC_IN_BOUNDS(kSiteEntry, base + (uint32_t)lane, ix.list_off[ix.lists]))
            id = __ldg(ix.ids + base + lane);
        if (!HC_IN_BOUNDS(kSiteRow, id, ix.rows)) id = 0;
    };
    auto issue = [&](uint32_t id, uint32_t cnt, uint32_t gi, uint32_t v, uint32_t stage) {
        const uint32_t col = s + v * LPR;
        const uint8_t* at = db + col * 16;
        const uint32_t to = slot + stage * 4096;
#pragma unroll
        for (int j = 0; j < G; ++j) {
            const uint32_t r = (gi * G + (uint32_t)j) * RPI + g;
            const uint32_t rid = __shfl_sync(0xffffffffu, id, (int)r);
            if (r < cnt && col < vecs) cp_async16(to + 512u * (uint32_t)j, at + (size_t)rid * row_bytes);
        }
    };
    uint32_t id, cnt, nid, ncnt, stage = 0;
    next_step(id, cnt);
    if (cnt == 0) return;
    issue(id, cnt, 0, 0, 0);
    cp_async_commit();
    next_step(nid, ncnt);
    while (cnt) {
        uint32_t fid = 0, fcnt = 0;
        if (ncnt) next_step(fid, fcnt);
#pragma unroll 1
        for (uint32_t gi = 0; gi < (uint32_t)NG; ++gi) {
            Acc part[G];
#pragma unroll
            for (int j = 0; j < G; ++j) part[j] = Acc(0);
#pragma unroll 1
            for (uint32_t v = 0; v < vpl; ++v) {
                // the unit after this one: this row part, this step or the next
                const bool same = v + 1 < vpl, step = !same && gi + 1 == (uint32_t)NG;
                issue(step ? nid : id, step ? ncnt : cnt, same ? gi : (step ? 0u : gi + 1),
                      same ? v + 1 : 0u, stage ^ 1u);
                cp_async_commit();
                const uint32_t col = s + v * LPR;
                const bool colok = col < vecs;
                const uint4 qv =
                    v == 0 ? qv0 : (colok ? ldg16(qrow + col * 16) : make_uint4(0, 0, 0, 0));
                cp_async_wait<1>();
                const uint8_t* from = ring + stage * 4096 + lane * 16;
#pragma unroll
                for (int j = 0; j < G; ++j) {
                    uint4 rv = *reinterpret_cast<const uint4*>(from + 512 * j);
                    if (!colok) rv = make_uint4(0, 0, 0, 0);
                    part[j] = acc_vec(rv, qv, part[j]);
                }
                stage ^= 1u;
            }
            // halving steps over the top log2(G) bits of s, then plain sums
#pragma unroll
            for (int w = LPR / 2, half = G / 2; half >= 1; w >>= 1, half >>= 1) {
                const bool upper = (s & (uint32_t)w) != 0;
#pragma unroll
                for (int t = 0; t < half; ++t) {
                    const Acc send = upper ? part[t] : part[t + half];
                    const Acc keep = upper ? part[t + half] : part[t];
                    part[t] = keep + __shfl_xor_sync(0xffffffffu, send, w);
                }
            }
            Acc dsum = part[0];
#pragma unroll
            for (int w = COPIES / 2; w >= 1; w >>= 1)
                dsum += __shfl_xor_sync(0xffffffffu, dsum, w);
            const uint32_t r = (gi * G + s / COPIES) * RPI + g;
            const uint32_t cid = __shfl_sync(0xffffffffu, id, (int)r);
            top.offer(r < cnt && (s % COPIES) == 0 ? ((uint64_t)dist_bits(dsum) << 32) | cid
                                                   : kEmpty,
                      k, lane);
        }
        id = nid, cnt = ncnt;
        nid = fid, ncnt = fcnt;
    }
    cp_async_wait<0>();
}

// ring: kRingRows rows of the warp's shared memory (rows of at most 128 bytes) or
// kWideRing bytes; SPLIT: steps part, part + parts, ... only; START as in
// StagedSteps, LATE as in walk_staged.  ROWS: kFullRows for rows of exactly 16 LPR bytes, kShortRows for
// shorter ones, kAnyRows where one kernel serves both (a kernel of its own for
// each spares registers: with both in one, 96-byte rows at k = 100 spilled, 5.2 against
// 4.6 ms for 60,000 queries at p = 200).
enum RowForm { kAnyRows, kFullRows, kShortRows };

template <bool F32, int LPR, int KR, bool SPLIT, bool START, int ROWS = kAnyRows,
          bool LATE = false>
__device__ __forceinline__ void walk_packed(const IndexView& ix, const uint8_t* qrow, uint32_t k,
                                            const uint32_t* win_at, const uint32_t* win_pre,
                                            uint32_t nm, uint32_t total, uint32_t part,
                                            uint32_t parts, uint8_t* ring, WarpTopK<KR>& top,
                                            int lane) {
    if constexpr (LPR > 8) {
        walk_wide<F32, LPR, KR, SPLIT>(ix, qrow, k, win_at, win_pre, nm, total, part, parts, ring,
                                       top, lane);
    } else if (ROWS == kFullRows || (ROWS == kAnyRows && ix.row_bytes == 16 * LPR)) {
        walk_staged<F32, LPR, KR, true, SPLIT, START, LATE>(ix, qrow, k, win_at, win_pre, nm, total,
                                                            part, parts, ring, top, lane);
    } else {
        walk_staged<F32, LPR, KR, false, SPLIT, START, LATE>(ix, qrow, k, win_at, win_pre, nm,
                                                             total, part, parts, ring, top, lane);
    }
}

// Algorithm 2 for one query over the lists L0, L0 + Lstep, ... into the warp's
// running top-k: positions, packed windows, then their walk.  pos_w, win_pre:
// one word per list of the index.
template <bool F32, int LPR, int KR, bool START = false, int ROWS = kAnyRows, bool LATE = false>
__device__ __forceinline__ void search_lists(const IndexView& ix, const uint8_t* qrow,
                                             uint32_t depth, uint32_t k, uint32_t L0,
                                             uint32_t Lstep, uint32_t* pos_w, uint32_t* win_pre,
                                             uint8_t* ring, WarpTopK<KR>& top, int lane,
                                             const int64_t* pos_in = nullptr,
                                             const uint32_t* pos_cm = nullptr) {
    load_positions(ix, qrow, pos_w, lane, L0, Lstep, pos_in, pos_cm);
    const uint32_t nm = ix.lists > L0 ? (ix.lists - L0 + Lstep - 1) / Lstep : 0;
    uint32_t* win_at = pos_w;   // positions are consumed by pack_windows
    const uint32_t total = pack_windows(ix, depth, L0, Lstep, pos_w, win_at, win_pre, lane);
    walk_packed<F32, LPR, KR, false, START, ROWS, LATE>(ix, qrow, k, win_at, win_pre, nm, total, 0,
                                                        1, ring, top, lane);
}

// The walk of a query's packed windows in the order of the row ids, kSweep
// entries at a time (a sweep): the ids of a sweep are sorted into 256 buckets of
// row ranges (a counting sort in shared memory) before its rows are read.  The
// warps of a block start every sweep together, so that at any time the SM reads
// rows of a small part of the database, whatever order the lists hold them in.
// counts: 256 words, sorted: kSweep words per warp.  Every warp of the block
// calls this, with total = 0 when it has no query.
constexpr int kSweepLoads = 32;
constexpr uint32_t kSweep = 32 * kSweepLoads;

template <bool F32, int LPR, int KR, bool FULL>
__device__ __forceinline__ void walk_sweeps(const IndexView& ix, const uint8_t* qrow, uint32_t k,
                                            const uint32_t* win_at, const uint32_t* win_pre,
                                            uint32_t nm, uint32_t total, uint32_t shift,
                                            uint32_t* counts, uint32_t* sorted, uint8_t* ring,
                                            WarpTopK<KR>& top, int lane) {
    StagedSteps<F32, LPR, KR, FULL, true> pipe(ix, qrow, ring, top, k);
    WindowCursor cur;
    const uint32_t sweeps = total / kSweep + (total % kSweep != 0);
    for (uint32_t s = 0; __syncthreads_or(s < sweeps); ++s) {
        if (s >= sweeps) continue;
        const uint32_t e0 = s * kSweep, cnt = min(kSweep, total - e0);
        uint32_t id[kSweepLoads];
#pragma unroll
        for (int u = 0; u < kSweepLoads; ++u)
            id[u] = cur.id(ix, win_at, win_pre, nm, total,
                           e0 + min(32 * (uint32_t)u + (uint32_t)lane, cnt - 1));
#pragma unroll
        for (int j = 0; j < 8; ++j) counts[32 * j + lane] = 0;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < kSweepLoads; ++u)
            if (32 * (uint32_t)u + (uint32_t)lane < cnt) atomicAdd(&counts[id[u] >> shift], 1u);
        __syncwarp();
        // exclusive prefixes: lane l owns buckets 8 l .. 8 l + 7
        uint4 lo4 = reinterpret_cast<const uint4*>(counts)[2 * lane];
        uint4 hi4 = reinterpret_cast<const uint4*>(counts)[2 * lane + 1];
        const uint32_t sum = lo4.x + lo4.y + lo4.z + lo4.w + hi4.x + hi4.y + hi4.z + hi4.w;
        uint32_t run = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += y;
        }
        run -= sum;
        uint4 a, b;
        a.x = run, a.y = a.x + lo4.x, a.z = a.y + lo4.y, a.w = a.z + lo4.z;
        b.x = a.w + lo4.w, b.y = b.x + hi4.x, b.z = b.y + hi4.y, b.w = b.z + hi4.z;
        reinterpret_cast<uint4*>(counts)[2 * lane] = a;
        reinterpret_cast<uint4*>(counts)[2 * lane + 1] = b;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < kSweepLoads; ++u)
            if (32 * (uint32_t)u + (uint32_t)lane < cnt)
                sorted[atomicAdd(&counts[id[u] >> shift], 1u)] = id[u];
        __syncwarp();
        for (uint32_t o = 0; o < cnt; o += 32) {
            const uint32_t n = min(32u, cnt - o);
            pipe.add(sorted[o + min((uint32_t)lane, n - 1)], n, top, k, lane, [] {});
        }
    }
    pipe.finish(top, k, lane);
}

}  // namespace hc
