// The walk of a batch in key order over a database larger than an SM's address
// translation reaches: rows read in sweeps of ascending ids.
#include "hc_walk.cuh"

namespace hc {

namespace {

// The walk on the positions of a batch search, rows read in sweeps of ascending
// ids (walk_sweeps; rows of at most 128 bytes): per warp a ring, the sweep's
// counters and sorted ids, and the positions.  shift: row id >> shift < 256.
// Words of a warp behind the rings, a multiple of four: the counters are read as
// 16-byte vectors.
__host__ __device__ __forceinline__ uint32_t sweep_words(uint32_t lists) {
    return 256 + kSweep + ((2 * lists + 3) & ~3u);
}

template <bool F32, int LPR, int KR>
__global__ void __launch_bounds__(kQWarps * 32, 2) sweep_kernel(QueryArgs a, uint32_t shift) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t w = blockIdx.x * kQWarps + warp;
    const IndexView& ix = a.ix;
    uint32_t qi = w < a.nq ? __ldg(a.order + w) : 0u;
    const bool mine = w < a.nq && HC_IN_BOUNDS(kSiteQuery, qi, a.nq);
    if (!mine) qi = 0;   // takes part in the block's barriers only
    const uint8_t* qrow = static_cast<const uint8_t*>(a.q) + (size_t)qi * ix.row_bytes;
    const uint32_t rb = ring_bytes<LPR>(ix.row_bytes);
    uint8_t* ring = smem + warp * rb;
    uint32_t* counts = reinterpret_cast<uint32_t*>(smem + kQWarps * rb) +
                       warp * sweep_words(ix.lists);
    uint32_t* sorted = counts + 256;
    uint32_t* pos_w = sorted + kSweep;
    uint32_t* win_pre = pos_w + ix.lists;
    WarpTopK<KR> top;
    top.init();
    uint32_t total = 0;
    if (mine) {
        load_positions(ix, qrow, pos_w, lane, 0, 1, nullptr, a.pos_cm + (size_t)qi * ix.lists);
        total = pack_windows(ix, a.p, 0, 1, pos_w, pos_w, win_pre, lane);
    }
    if (ix.row_bytes == 16 * LPR)
        walk_sweeps<F32, LPR, KR, true>(ix, qrow, a.k, pos_w, win_pre, ix.lists, total, shift,
                                        counts, sorted, ring, top, lane);
    else
        walk_sweeps<F32, LPR, KR, false>(ix, qrow, a.k, pos_w, win_pre, ix.lists, total, shift,
                                         counts, sorted, ring, top, lane);
    if (mine)
        top.template store<F32>(a.k, lane, a.out_ids + (size_t)qi * a.k,
                                static_cast<uint32_t*>(a.out_dist) + (size_t)qi * a.k);
}

template <bool F32, int LPR, int KR>
struct SweepLaunch {
    static size_t shared(uint32_t row_bytes, uint32_t lists) {
        return kQWarps * (ring_bytes<LPR>(row_bytes) + sizeof(uint32_t) * sweep_words(lists));
    }
    static cudaError_t run(const QueryArgs& a, cudaStream_t s) {
        if constexpr (!F32 && LPR <= 8 && KR != 4) {
            const size_t smem = shared(a.ix.row_bytes, a.ix.lists);
            const cudaError_t e =
                allow_shared(sweep_kernel<F32, LPR, KR>, shared(16 * LPR, kMaxLists));
            if (e != cudaSuccess) return e;
            uint32_t shift = 0;
            while ((a.ix.rows - 1) >> shift > 255) ++shift;
            const unsigned blocks = (unsigned)(((uint64_t)a.nq + kQWarps - 1) / kQWarps);
            sweep_kernel<F32, LPR, KR><<<blocks, kQWarps * 32, smem, s>>>(a, shift);
            count_launches(1);
            return cudaGetLastError();
        } else {
            return cudaErrorInvalidValue;   // walk_kind: uint8 rows of at most 128 bytes, k <= 64
        }
    }
};

}  // namespace

cudaError_t launch_sweeps(const QueryArgs& a, cudaStream_t s) {
    return dispatch<SweepLaunch>(a.ix.P.dtype == HC_F32, lanes_per_row(a.ix.row_bytes),
                                 regs_for_k(a.k), a, s);
}

}  // namespace hc
