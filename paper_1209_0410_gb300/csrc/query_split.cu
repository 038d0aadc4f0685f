// Small batches in arrival order: several warps to a query, so that a handful of
// queries occupies the chip and a single one does not wait on a serial walk.
// Bound by latency: the launch, two rounds of dependent loads for the key, four
// or five for the search, then 1/16 of the steps (100,000 rows, p = 128: one query
// repeated 20 us against 56 with one warp, a query not seen before 76 against 110 with
// the first touch of its lines; 1,000 queries at p = 64: 34 against 47 us).
// Batches of other streams fill the time a block waits: three blocks of 8 warps fit
// an SM beside each other.  Blocks of 16 with 128 registers, one per SM, left 320
// batches of 400 queries on 16 streams at 4.8 ms (p = 64; 2.2 ms now, 2.1 with a warp
// per query); they stay where a query takes all 16.
#include "hc_walk.cuh"

namespace hc {

namespace {

// A small batch: wpq warps (a power of two up to W, the warps of a block) share a
// query.  They search its lists with their lanes spread over the probes, walk every
// wpq-th step each and merge their lists pairwise.  BLOCKS: blocks resident per SM.
template <bool F32, int LPR, int KR, int W, int BLOCKS, int ROWS>
__global__ void __launch_bounds__(W * 32, BLOCKS) split_kernel(QueryArgs a, uint32_t wpq) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t group = warp / wpq, sub = warp % wpq;
    const uint32_t qi = blockIdx.x * (W / wpq) + group;
    const bool mine = qi < a.nq;   // the others only take part in the barriers
    const IndexView& ix = a.ix;
    const uint8_t* qrow = static_cast<const uint8_t*>(a.q) + (size_t)(mine ? qi : 0) * ix.row_bytes;
    const uint32_t rb = ring_bytes<LPR>(ix.row_bytes);
    uint64_t* lists = reinterpret_cast<uint64_t*>(smem + W * rb);
    uint64_t* list = lists + (size_t)warp * 32 * KR;
    uint32_t* totals = reinterpret_cast<uint32_t*>(lists + W * 32 * KR);
    uint32_t* pos_w = totals + W + group * 2 * ix.lists;
    uint32_t* win_pre = pos_w + ix.lists;
    // the query's keys, by one of its warps, in that warp's ring
    ulonglong2* keys = reinterpret_cast<ulonglong2*>(smem + group * wpq * rb);
    if (!a.pos_in) {
        if (mine && sub == 0 && (uint32_t)lane < ix.P.curves) {
            uint64_t hi, lo;
            curve_key_call(qrow, ix.P, (uint32_t)lane, hi, lo);
            keys[lane] = make_ulonglong2(hi, lo);
        }
        __syncthreads();
        if (mine) query_positions_spread(ix, keys, pos_w, lane, sub, wpq);
    } else if (mine) {
        load_positions(ix, qrow, pos_w, lane, sub, wpq, a.pos_in + (size_t)qi * ix.lists, nullptr);
    }
    __syncthreads();
    if (mine && sub == 0) {
        const uint32_t depth = a.p_query ? __ldg(a.p_query + qi) : a.p;
        const uint32_t total = pack_windows(ix, depth, 0, 1, pos_w, pos_w, win_pre, lane);
        if (lane == 0) totals[group] = total;
    }
    __syncthreads();
    WarpTopK<KR> top;
    top.init();
    constexpr bool kStart = LPR <= 8 && (BLOCKS < 3 || KR == 1 || LPR < 8);
    if (mine)
        walk_packed<F32, LPR, KR, true, kStart, ROWS>(ix, qrow, a.k, pos_w, win_pre, ix.lists,
                                                      totals[group], sub, wpq, smem + warp * rb,
                                                      top, lane);
#pragma unroll
    for (int r = 0; r < KR; ++r) list[r * 32 + lane] = top.v[r];
    for (uint32_t step = 1; step < wpq; step *= 2) {
        __syncthreads();
        if (sub % (2 * step) == 0)
            merge_lists<KR>(list, list + (size_t)step * 32 * KR, a.k, lane);
    }
    if (mine && sub == 0) {
#pragma unroll
        for (int r = 0; r < KR; ++r) top.v[r] = list[r * 32 + lane];
        top.template store<F32>(a.k, lane, a.out_ids + (size_t)qi * a.k,
                                static_cast<uint32_t*>(a.out_dist) + (size_t)qi * a.k);
    }
}

template <bool F32, int LPR, int KR>
struct SplitLaunch {
    // W: warps, per: queries of a block
    static size_t shared(uint32_t row_bytes, uint32_t lists, uint32_t W, uint32_t per) {
        return W * (ring_bytes<LPR>(row_bytes) + 256 * KR + 4) + 8ull * per * lists;
    }
    template <int W, int BLOCKS, int ROWS>
    static cudaError_t go(const QueryArgs& a, uint32_t wpq, cudaStream_t s) {
        auto kernel = split_kernel<F32, LPR, KR, W, BLOCKS, ROWS>;
        const uint32_t per = W / wpq;
        const cudaError_t e = allow_shared(kernel, shared(16 * LPR, kMaxLists, W, W / 2));
        if (e != cudaSuccess) return e;
        kernel<<<(a.nq + per - 1) / per, W * 32, shared(a.ix.row_bytes, a.ix.lists, W, per), s>>>(
            a, wpq);
        count_launches(1);
        return cudaGetLastError();
    }
    static cudaError_t run(const QueryArgs& a, uint32_t wpq, cudaStream_t s) {
        if constexpr (KR == 2) {
            return cudaErrorInvalidValue;   // launch_split takes 4
        } else {
            if (wpq > (uint32_t)kSplitBlock) return go<kSplitWarps, 1, kAnyRows>(a, wpq, s);
            if constexpr (LPR <= 8)
                if (a.ix.row_bytes == 16 * LPR)
                    return go<kSplitBlock, 3, kFullRows>(a, wpq, s);
            return go<kSplitBlock, 3, LPR <= 8 ? kShortRows : kAnyRows>(a, wpq, s);
        }
    }
};

}  // namespace

cudaError_t launch_split(const QueryArgs& a, uint32_t wpq, cudaStream_t s) {
    return dispatch<SplitLaunch>(a.ix.P.dtype == HC_F32, lanes_per_row(a.ix.row_bytes),
                                 a.k <= 32 ? 1 : 4, a, wpq, s);
}

}  // namespace hc
