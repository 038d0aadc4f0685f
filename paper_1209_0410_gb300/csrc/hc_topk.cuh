// Warp-wide running top-k over packed candidates (FindTopK of Sec. 5.1 and
// the Aggregator's reduction of Sec. 4.1 in one structure).
//
// A candidate is the 64-bit value (distance bits << 32) | id, so ascending
// packed order is ascending (distance, id): ties go to the lower id.  uint8
// distances are non-negative int32; float32 distances are non-negative
// floats, whose bit patterns order like the values.  ~0 marks an empty slot
// and sorts after every real candidate.
//
// The list is kept sorted across the warp: element e = r*32 + lane lives in
// register r of that lane, KR registers per lane (k <= 32*KR).  A batch of 32
// candidates (one per lane) is filtered against the k-th element; survivors
// are inserted one at a time with a ballot rank and a one-slot shuffle.  An
// id already in the list has an identical packed value (same row, same
// query), so an equal value is dropped: that is the de-duplication of
// candidates returned by several curves or windows.
#pragma once

#include <stdint.h>

namespace hc {

constexpr uint64_t kEmpty = ~0ull;

// Bitonic compare-exchange steps over 32 KR entries, entry r 32 + lane in v[r]
// of the lane.  merge_sorted: the last phase alone (a bitonic sequence in,
// ascending out); sort_all: any order in.
template <int KR>
__device__ __forceinline__ void bitonic_phase(uint64_t (&v)[KR], int size, int stride, int lane) {
    if (stride >= 32) {
        const int rs = stride / 32;
#pragma unroll
        for (int r = 0; r < KR; ++r) {
            if ((r & rs) == 0) {
                const bool up = ((r * 32) & size) == 0;   // size > 32 here
                const uint64_t lo = min(v[r], v[r | rs]), hi = max(v[r], v[r | rs]);
                v[r] = up ? lo : hi;
                v[r | rs] = up ? hi : lo;
            }
        }
    } else {
#pragma unroll
        for (int r = 0; r < KR; ++r) {
            const uint64_t o = __shfl_xor_sync(0xffffffffu, v[r], stride);
            const bool up = ((r * 32 + lane) & size) == 0, first = (lane & stride) == 0;
            v[r] = (first == up) ? min(v[r], o) : max(v[r], o);
        }
    }
}
template <int KR>
__device__ __forceinline__ void merge_sorted(uint64_t (&v)[KR], int lane) {
#pragma unroll
    for (int stride = 16 * KR; stride >= 1; stride >>= 1)
        bitonic_phase<KR>(v, 64 * KR, stride, lane);
}
template <int KR>
__device__ __forceinline__ void sort_all(uint64_t (&v)[KR], int lane) {
#pragma unroll
    for (int size = 2; size <= 32 * KR; size <<= 1)
#pragma unroll
        for (int stride = size / 2; stride >= 1; stride >>= 1)
            bitonic_phase<KR>(v, size, stride, lane);
}

// the warp's 32 values in order (out of line: one copy per translation unit)
static __device__ __noinline__ uint64_t sort_warp(uint64_t x, int lane) {
    uint64_t v[1] = {x};
    sort_all<1>(v, lane);
    return v[0];
}

template <int KR>
struct WarpTopK {
    uint64_t v[KR];

    __device__ __forceinline__ void init() {
#pragma unroll
        for (int r = 0; r < KR; ++r) v[r] = kEmpty;
    }

    // element k-1 (warp-uniform result)
    __device__ __forceinline__ uint64_t kth(uint32_t k) const {
        const uint32_t e = k - 1, rr = e >> 5;
        uint64_t x = v[0];
#pragma unroll
        for (int r = 1; r < KR; ++r)
            if ((uint32_t)r == rr) x = v[r];
        return __shfl_sync(0xffffffffu, x, (int)(e & 31));
    }

    __device__ __forceinline__ void insert(uint64_t y, int lane) {
        uint32_t pos = 0;
        bool dup = false;
#pragma unroll
        for (int r = 0; r < KR; ++r) {
            pos += __popc(__ballot_sync(0xffffffffu, v[r] < y));
            dup |= __any_sync(0xffffffffu, v[r] == y) != 0;
        }
        if (dup) return;
#pragma unroll
        for (int r = KR - 1; r >= 0; --r) {
            const uint64_t up = __shfl_up_sync(0xffffffffu, v[r], 1);
            uint64_t carry = kEmpty;
            if (r > 0) carry = __shfl_sync(0xffffffffu, v[r > 0 ? r - 1 : 0], 31);
            const uint64_t prev = lane == 0 ? carry : up;
            const uint32_t e = (uint32_t)r * 32 + lane;
            v[r] = e > pos ? prev : (e == pos ? y : v[r]);
        }
    }

    // offer one candidate per lane
    __device__ __forceinline__ void offer(uint64_t cand, uint32_t k, int lane) {
        uint64_t thr = kth(k);
        uint32_t m = __ballot_sync(0xffffffffu, cand < thr);
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            const uint64_t y = __shfl_sync(0xffffffffu, cand, src);
            if (y < thr) {
                insert(y, lane);
                thr = kth(k);
            }
        }
    }

    // one of 32 candidates as the very first: the list is the sorted candidates;
    // false (nothing done) when two of them are equal
    __device__ __forceinline__ bool start(uint64_t cand, int lane) {
        const uint64_t x = sort_warp(cand, lane);
        const uint64_t up = __shfl_up_sync(0xffffffffu, x, 1);
        if (__any_sync(0xffffffffu, lane > 0 && up == x && x != kEmpty)) return false;
        v[0] = x;
        return true;
    }

    // offer one row per lane: distance bits and id (live: the lane has one); thr:
    // the k-th element, kept by the caller.  The first test is on the distance
    // bits alone.
    __device__ __forceinline__ void offer_row(uint32_t dist, uint32_t id, bool live, uint32_t k,
                                              uint64_t& thr, int lane) {
        uint32_t m = __ballot_sync(0xffffffffu, live && dist <= (uint32_t)(thr >> 32));
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            const uint64_t y = ((uint64_t)__shfl_sync(0xffffffffu, dist, src) << 32) |
                               __shfl_sync(0xffffffffu, id, src);
            if (y < thr) {
                insert(y, lane);
                thr = kth(k);
            }
        }
    }

    // results e < k: ids (-1 for empty) and distances (empty -> int32 max or +inf)
    template <bool F32>
    __device__ __forceinline__ void store(uint32_t k, int lane, int32_t* ids, void* dist) const {
#pragma unroll
        for (int r = 0; r < KR; ++r) {
            const uint32_t e = (uint32_t)r * 32 + lane;
            if (e < k) {
                const uint64_t x = v[r];
                const bool empty = x == kEmpty;
                ids[e] = empty ? -1 : (int32_t)(uint32_t)x;
                const uint32_t dbits = (uint32_t)(x >> 32);
                if (F32)
                    static_cast<uint32_t*>(dist)[e] = empty ? 0x7F800000u : dbits;
                else
                    static_cast<int32_t*>(dist)[e] = empty ? 0x7FFFFFFF : (int32_t)dbits;
            }
        }
    }
};

// Sorted list `other` into sorted list `mine`, both 32 KR words of shared memory
// with distinct elements each, by one warp: the k smallest distinct of the two
// lead `mine` afterwards.  With k <= 16 KR the smaller of element e of one and
// 32 KR - 1 - e of the other are a bitonic sequence of the 32 KR smallest, which
// hold k distinct ones; otherwise `other` is offered to `mine`.  Out of line.
template <int KR>
static __device__ __noinline__ void merge_lists(uint64_t* mine, const uint64_t* other, uint32_t k,
                                                int lane) {
    WarpTopK<KR> top;
#pragma unroll
    for (int r = 0; r < KR; ++r) top.v[r] = mine[r * 32 + lane];
    if (k > 16 * KR) {
#pragma unroll 1
        for (int r = 0; r < KR; ++r) top.offer(other[r * 32 + lane], k, lane);
    } else {
#pragma unroll
        for (int r = 0; r < KR; ++r)
            top.v[r] = min(top.v[r], other[32 * KR - 1 - (r * 32 + lane)]);
        merge_sorted<KR>(top.v, lane);
        bool twice[KR], any = false;
#pragma unroll
        for (int r = 0; r < KR; ++r) {
            const uint64_t up = __shfl_up_sync(0xffffffffu, top.v[r], 1);
            const uint64_t before = __shfl_sync(0xffffffffu, top.v[r > 0 ? r - 1 : 0], 31);
            const uint64_t prev = lane ? up : (r > 0 ? before : kEmpty);
            twice[r] = top.v[r] == prev && top.v[r] != kEmpty;
            any |= twice[r];
        }
        if (__any_sync(0xffffffffu, any)) {
#pragma unroll
            for (int r = 0; r < KR; ++r)
                if (twice[r]) top.v[r] = kEmpty;
            sort_all<KR>(top.v, lane);
        }
    }
#pragma unroll
    for (int r = 0; r < KR; ++r) mine[r * 32 + lane] = top.v[r];
    __syncwarp();
}

}  // namespace hc
