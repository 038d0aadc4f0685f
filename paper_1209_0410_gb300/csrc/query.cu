// K3..K6: the fused query kernel (Algorithm 2 for a batch of queries); the
// exact brute-force kNN (Eq. 3), which shares its distance and top-k code,
// is in brute.cu.
//
// One warp per query:
//   K1  lanes c < curves compute the query's extended-key on curve c;
//   K3  lanes L < lists run lower_bound in list L (128-bit compares; the low
//       word is consulted only when the high words tie, recomputed from the
//       entry's row when the index keeps high words only), starting on the
//       index's fence of every 16th high word.  For hc_query_ordered, K1 and
//       K3 run before the walk as passes over the whole batch instead
//       (order_keys_kernel: every curve's key of every query; a sort by each
//       curve's key; batch_positions_kernel: a warp per 32 neighbouring keys
//       of one curve), and the walk reads the positions;
//   K4  the windows [max(0,pos-p), min(n,pos+p)) are packed back to back and
//       walked 32 entries at a time (a step may span several).  Rows of at most
//       128 bytes are staged: the next step's rows are copied into a two-step
//       per-warp shared-memory ring with cp.async while the current step is
//       reduced, so the bytes in flight are bounded by shared memory instead of
//       registers, and each lane then reads a whole row (16-byte vectors laid
//       out so that no two lanes of a quarter-warp meet in a bank): no partial
//       sums cross lanes.  Wider rows go through a ring of two 4 KB units, LPR
//       lanes to a row and eight 16-byte vectors per lane and unit, and are
//       reduce-scattered over the LPR lanes.  uint8 distances use vabsdiffu4 + dp4a (exact in
//       32-bit integers), float32 use fma;
//   K5/K6 the 32 packed (distance, id) candidates are offered to one running
//       warp top-k for the whole query, which drops duplicate ids: the union
//       over curves and partitions and the Aggregator's reduction in one.
// The path is a gather bounded by HBM bandwidth; no tensor cores are used.
#include <algorithm>

#include "hc_walk.cuh"

namespace hc {

namespace {

// Rows of at most 128 bytes go through a two-step cp.async ring in shared
// memory: the block's rings, then its positions and window prefixes.
// BLOCKS: blocks resident per SM (registers)
template <bool F32, int LPR, int KR, int BLOCKS, int ROWS, bool LATE = false>
__global__ void __launch_bounds__(kQWarps * 32, BLOCKS) query_kernel(QueryArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t w = blockIdx.x * kQWarps + warp;
    if (w >= a.nq) return;
    const uint32_t qi = a.order ? __ldg(a.order + w) : w;
    if (!HC_IN_BOUNDS(kSiteQuery, qi, a.nq)) return;
    const IndexView& ix = a.ix;
    const uint8_t* qrow = static_cast<const uint8_t*>(a.q) + (size_t)qi * ix.row_bytes;
    const uint32_t depth = a.p_query ? __ldg(a.p_query + qi) : a.p;
    const uint32_t rb = ring_bytes<LPR>(ix.row_bytes);
    uint32_t* pos_w = reinterpret_cast<uint32_t*>(smem + kQWarps * rb) + warp * 2 * ix.lists;
    WarpTopK<KR> top;
    top.init();
    constexpr bool kStart = LPR <= 8 && (BLOCKS == 2 || KR == 1 || LPR < 8);
    search_lists<F32, LPR, KR, kStart, ROWS, LATE>(
        ix, qrow, depth, a.k, 0, 1, pos_w, pos_w + ix.lists, smem + warp * rb, top, lane,
        a.pos_in ? a.pos_in + (size_t)qi * ix.lists : nullptr,
        a.pos_cm ? a.pos_cm + (size_t)qi * ix.lists : nullptr);
    top.template store<F32>(a.k, lane, a.out_ids + (size_t)qi * a.k,
                            static_cast<uint32_t*>(a.out_dist) + (size_t)qi * a.k);
}

// keys[c nq + i] = top kOrderBits bits of query i's curve-c extended-key
// for c < ncurves; with qhi / qlo, also the key's two words.  One thread per
// query: 16-coordinate curves of consecutive dimensions four at a time as
// byte lanes of 32-bit words (as the build's key pass), others one by one.
__device__ __forceinline__ void put_order_key(const IndexView& ix, uint32_t nq, uint32_t i,
                                              uint32_t c, uint64_t h, uint64_t l, uint64_t* keys,
                                              uint64_t* qhi, uint64_t* qlo) {
    const size_t t = (size_t)c * nq + i;
    const uint32_t bits = 8 * ix.P.m;   // key bits, right-aligned in (h, l)
    const uint64_t top = bits > 64 ? (h << (128 - bits)) | (bits < 128 ? l >> (bits - 64) : 0)
                                   : l << (64 - bits);
    keys[t] = top >> (64 - kOrderBits);
    if (qhi) {
        qhi[t] = h;
        qlo[t] = l;
    }
}

__global__ void __launch_bounds__(256) order_keys_kernel(IndexView ix, const uint8_t* q,
                                                         uint32_t nq, uint32_t ncurves,
                                                         uint64_t* keys, uint64_t* qhi,
                                                         uint64_t* qlo) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nq) return;
    const uint8_t* row = q + (size_t)i * ix.row_bytes;
    uint32_t c = 0;
    if (ix.P.m == 16 && ix.P.dim_map == nullptr) {
        for (; c + 4 <= ncurves; c += 4) {
            uint4 cb[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) cb[t] = curve_bytes16(row, ix.P.dtype, c + t);
            uint64_t hi[4], lo[4];
            hilbert_keys4<false>(cb, hi, lo);
#pragma unroll
            for (int t = 0; t < 4; ++t) put_order_key(ix, nq, i, c + t, hi[t], lo[t], keys, qhi, qlo);
        }
    }
    for (; c < ncurves; ++c) {
        uint64_t h, l;
        curve_key_call(row, ix.P, c, h, l);
        put_order_key(ix, nq, i, c, h, l, keys, qhi, qlo);
    }
}

// searches a lane of batch_positions_kernel runs side by side (1, 2 and 8
// measured slower on 32 partitions)
constexpr int kBatchILP = 4;

// at[0 .. G) to p[0 .. G), p aligned to 4 G bytes
template <int G>
__device__ __forceinline__ void store_group(uint32_t* p, const uint32_t (&at)[G]) {
    if constexpr (G == 4) {
        *reinterpret_cast<uint4*>(p) = make_uint4(at[0], at[1], at[2], at[3]);
    } else if constexpr (G == 2) {
        *reinterpret_cast<uint2*>(p) = make_uint2(at[0], at[1]);
    } else {
#pragma unroll
        for (int g = 0; g < G; ++g) p[g] = at[g];
    }
}

// Queries a lane of batch_positions_kernel takes: kBatchILP searches side by
// side are kBatchILP partitions of one query (three partitions or more: the
// last group may be partial), or the partitions of four queries (one
// partition) or of two (two partitions).
__host__ __device__ __forceinline__ uint32_t batch_queries_per_lane(uint32_t parts) {
    return parts == 1 ? 4u : (parts == 2 ? 2u : 1u);
}
static_assert(kBatchILP == 4, "queries per lane assume four searches side by side");

// K3 for a whole batch.  Warp w takes curve c = w / tiles and tile t = w %
// tiles: the 32 qpl queries at ranks 32 qpl t .. of curve c's key order, lane
// l the ranks 32 qpl t + 32 u + l (u < qpl, qpl queries per lane).  Each lane
// searches its queries' curve-c keys in list j * curves + c of every
// partition j and writes the position to pos[query][c * partitions + j].  The
// 32 keys of a warp's round are neighbours on curve c, so the lanes' probes
// fall on the same few lines (one request serves many lanes) where lanes of a
// per-query warp would each probe a different list.
template <int QPL>   // batch_queries_per_lane(partitions)
__global__ void __launch_bounds__(256) batch_positions_kernel(IndexView ix, uint32_t nq,
                                                              const uint32_t* __restrict__ order,
                                                              const uint64_t* __restrict__ qhi,
                                                              const uint64_t* __restrict__ qlo,
                                                              uint32_t* __restrict__ pos) {
    constexpr int G = kBatchILP;
    constexpr uint32_t qpl = QPL;
    const int lane = threadIdx.x & 31;
    const uint64_t w = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t curves = ix.P.curves, parts = ix.lists / curves;
    const uint32_t span = 32 * qpl;
    const uint32_t tiles = (uint32_t)(((uint64_t)nq + span - 1) / span);
    if (w >= (uint64_t)tiles * curves) return;
    const uint32_t c = (uint32_t)(w / tiles), t = (uint32_t)(w % tiles);
    // the lane's queries; lanes past the batch search with query 0's key and
    // write nothing
    uint32_t qi[QPL];
    bool live[QPL];
    uint64_t kh[QPL], kl[QPL];
#pragma unroll
    for (int u = 0; u < QPL; ++u) {
        const uint32_t r = t * span + (uint32_t)u * 32 + (uint32_t)lane;
        live[u] = r < nq;
        qi[u] = live[u] ? __ldg(order + (size_t)c * nq + r) : 0u;
        if (live[u] && !HC_IN_BOUNDS(kSiteQuery, qi[u], nq)) {
            live[u] = false;
            qi[u] = 0;
        }
        kh[u] = __ldg(qhi + (size_t)c * nq + qi[u]);
        kl[u] = __ldg(qlo + (size_t)c * nq + qi[u]);
    }
    uint32_t lists[G], at[G];
    bool on[G];
    uint64_t gh[G], gl[G];
    if constexpr (QPL > 1) {
        // one round: search g is partition g % (G / QPL) of query g / (G / QPL)
        constexpr int PP = G / QPL;   // partitions (1 or 2)
#pragma unroll
        for (int g = 0; g < G; ++g) {
            on[g] = live[g / PP];
            gh[g] = kh[g / PP];
            gl[g] = kl[g / PP];
            lists[g] = (uint32_t)(g % PP) * curves + c;
        }
        lower_bound_lists<G>(ix, lists, on, gh, gl, at);
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (on[g])
                pos[(size_t)qi[g / PP] * ix.lists + (size_t)c * PP + (uint32_t)(g % PP)] = at[g];
        return;
    }
    uint32_t* out = pos + (size_t)qi[0] * ix.lists + (size_t)c * parts;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        gh[g] = kh[0];
        gl[g] = kl[0];
    }
    // G partitions at a time: their searches share the key
    for (uint32_t j0 = 0; j0 < parts; j0 += G) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
            on[g] = j0 + g < parts;
            lists[g] = on[g] ? (j0 + g) * curves + c : 0u;
        }
        lower_bound_lists<G>(ix, lists, on, gh, gl, at);
        if (!live[0]) continue;
        if (parts % G == 0) {
            // whole groups: one vector store (the row offset is a multiple
            // of the group since partitions are)
            store_group(out + j0, at);
        } else {
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (on[g]) out[j0 + g] = at[g];
        }
    }
}

__global__ void __launch_bounds__(kQWarps * 32) positions_kernel(QueryArgs a) {
    extern __shared__ uint32_t s_pos[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t qi = blockIdx.x * kQWarps + warp;
    if (qi >= a.nq) return;
    const uint8_t* qrow = static_cast<const uint8_t*>(a.q) + (size_t)qi * a.ix.row_bytes;
    uint32_t* pos_w = s_pos + warp * a.ix.lists;
    query_positions(a.ix, qrow, pos_w, lane);
    for (uint32_t L = lane; L < a.ix.lists; L += 32)
        a.out_pos[(size_t)qi * a.ix.lists + L] = (int64_t)pos_w[L];
}

// fence[j] = keys_hi[16 j] & kFenceMask: one thread per fence word
__global__ void __launch_bounds__(256) fence_kernel(const uint64_t* __restrict__ keys_hi,
                                                    uint64_t len, uint64_t* __restrict__ fence) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < len; j += stride)
        fence[j] = __ldg(keys_hi + (j << kFenceShift)) & kFenceMask;
}

// How a batch is walked (walk_kind).
enum Walk { kPlain, kLate, kByPartition, kSweeps };

template <bool F32, int LPR, int KR>
struct QueryLaunch {
    static size_t shared(uint32_t row_bytes, uint32_t lists) {
        return kQWarps * (ring_bytes<LPR>(row_bytes) + 2 * sizeof(uint32_t) * lists);
    }
    template <typename K>
    static cudaError_t go(K kernel, const QueryArgs& a, size_t smem, cudaStream_t s) {
        const cudaError_t e = allow_shared(kernel, shared(16 * LPR, kMaxLists));
        if (e != cudaSuccess) return e;
        const unsigned blocks = (unsigned)(((uint64_t)a.nq + kQWarps - 1) / kQWarps);
        kernel<<<blocks, kQWarps * 32, smem, s>>>(a);
        count_launches(1);
        return cudaGetLastError();
    }
    static cudaError_t run(const QueryArgs& a, Walk walk, cudaStream_t s) {
        const size_t smem = shared(a.ix.row_bytes, a.ix.lists);
        if constexpr (LPR <= 8) {
            const bool full = a.ix.row_bytes == 16 * LPR;
            if constexpr (!F32 && KR == 1)   // walk_kind: uint8, whole lines, k <= 32
                if (walk == kLate)
                    return go(query_kernel<F32, LPR, KR, 3, kFullRows, true>, a, smem, s);
            if constexpr (!F32 && KR != 4)   // walk_kind: uint8, k <= 64
                if (walk == kByPartition)
                    return full ? go(query_kernel<F32, LPR, KR, 2, kFullRows>, a, smem, s)
                                : go(query_kernel<F32, LPR, KR, 2, kShortRows>, a, smem, s);
            return full ? go(query_kernel<F32, LPR, KR, 3, kFullRows>, a, smem, s)
                        : go(query_kernel<F32, LPR, KR, 3, kShortRows>, a, smem, s);
        } else {
            return go(query_kernel<F32, LPR, KR, 3, kAnyRows>, a, smem, s);
        }
    }
};

int sm_count() {
    int sms = 152, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// The address translation of an SM reaches 256 MB (128 pages of 2 MB: 16 MB of
// random 128-byte rows, all in L2, arrive at 22 TB/s when they are spread over up to
// 256 MB, at 8.4 over 384 MB and at 5.7 over 1.2 GB).  A batch that fills the SMs several times over reads its
// rows of a larger database
//   kByPartition  when a partition's rows are within reach: the walk goes
//                 partition by partition as it is, and with 16 instead of 24
//                 warps per SM they stay in the same one (8 partitions of 160
//                 MB, 100,000 queries at p = 32: 4.2 against 6.3 ms, sweeps 4.6;
//                 8 of 128 MB, 60,000 queries, by window entries E: in key order
//                 E = 768 0.92 against 0.86, 2,048 1.50 against 1.58; in arrival
//                 order E = 512 1.27 against 1.52, 3,200 3.5 against 4.1);
//   kSweeps       in key order otherwise, sorted by row id (100,000 queries at p =
//                 128 on 10M rows: 2.5 against 3.9 ms; 20M 3.0 against 4.2, 50M 3.8
//                 against 4.4; 3M rows, 384 MB: 2.4 against 2.7; 1.5M rows, 192
//                 MB: 2.4 against 1.8, so the line lies between; 96-byte rows,
//                 which straddle lines, 384 MB: 1.41 against 1.32, 768 MB: 1.47
//                 against 1.72).  The sort of a sweep wants whole sweeps (60,000
//                 queries, 1 GB: E = 256 0.58 against 0.48 ms, 768 0.84 against
//                 0.99, but on 384 MB 0.83 against 0.75) and a short list (k = 37,
//                 E = 2,048: 2.6 against 2.4, 4,096 3.3 against 3.7; k = 100 is
//                 no faster).
// In arrival order the rows come from DRAM, which then binds (sweeps 4.6 against
// 4.2 ms), and rows wider than 128 bytes need fewer translations per byte.  3,000
// queries, one wave: 0.23 ms by partition, 0.20 plain; 12,000 gain as 60,000 do.
constexpr uint64_t kReachBytes = 320ull << 20, kReachStraddling = 512ull << 20;
constexpr uint64_t kReachPartition = 200ull << 20;

// A batch whose last wave is nearly full (full_waves) is done when its slowest warp
// is.  On rows at or past the reach, asking for the ids behind the next step's rows
// makes every walk of such a batch up to 11% shorter (k = 10, p = 300, 340 MB: 3,300
// queries 0.30 against 0.34 ms, 7,296 0.58 against 0.62); elsewhere asking before them is
// faster (4,000 to 6,000 queries 0 to 3%, 18,000 up to 9%, 128 MB 5 to 12%, depths that
// differ up to 11%).
constexpr uint64_t kLateBytes = 240ull << 20;

bool full_waves(uint64_t nq, uint64_t most) {
    const uint64_t wave = 3ull * kQWarps * sm_count();   // warps resident
    if (nq > most * wave) return false;
    const uint64_t last = nq % wave == 0 ? wave : nq % wave;
    return 100 * last >= (nq <= wave ? 66 : 80) * wave;
}

Walk walk_kind(const QueryArgs& a) {
    const IndexView& ix = a.ix;
    const uint64_t bytes = ix.rows * ix.row_bytes, parts = ix.lists / ix.P.curves;
    const bool whole_lines = (ix.row_bytes & (ix.row_bytes - 1)) == 0;
    if (ix.P.dtype == HC_U8 && (ix.row_bytes == 64 || ix.row_bytes == 128) && !a.order &&
        !a.p_query && a.k <= 32 && bytes / parts >= kLateBytes &&
        full_waves(a.nq, bytes / parts < kReachBytes ? 5 : 3))
        return kLate;
    if (ix.P.dtype != HC_U8 || ix.row_bytes > 128 || a.p_query ||
        bytes < (whole_lines ? kReachBytes : kReachStraddling) ||
        a.nq < 4ull * sm_count() * 2 * kQWarps)
        return kPlain;
    const uint64_t entries = 2ull * a.p * ix.lists;   // of a query's windows
    if (parts > 1 && bytes / parts < kReachPartition)
        return entries >= (!a.pos_cm ? 512 : a.k <= 32 ? 2048 : 4096) && a.k <= 64 ? kByPartition
                                                                                   : kPlain;
    // at most 96 lists: two blocks' shared memory per SM
    return a.pos_cm && ix.lists <= 96 && a.k <= 64 && entries >= (a.k <= 32 ? 1024 : 3200)
               ? kSweeps
               : kPlain;
}

// Warps per query when a batch in arrival order would leave SMs idle.
// Two as long as 16 warps per SM hold them (1,500 queries at two warps each took 83 us
// where 2,000 at one take 77), if the walk is worth a second search and a merge: 384
// entries (k = 10, 1,000 queries: 30 against 33 us), with the slower inserts of k > 32
// 4,096 (k = 33: 1,024 entries 91 against 72 us, 4,096 the same).
// Four and eight cost the chip 9 and 22 ns more per query, which a lone batch does not
// notice but batches on other streams do (16 streams, 400 queries each, p = 64: 26 ns
// per query at four, 17 at two).  So they are for batches that leave most of the chip
// free (6 to 8 warps per SM hold them; such a batch takes no longer than its launch by
// the host), and for walks on which they cost no more than 10%: 1,024 uint8 rows per
// warp (32 steps; 304 queries of 25,600 rows each: 106 us at eight, 150 at four; at half
// the rows, 400 queries on 16 streams run at 0.8 of a warp per query) or 128 KB of float32
// rows, or where each query has its own depth, so that the deepest sets the time (458
// queries at depths the predictor chose: 81 us at four warps, 111 at two).
uint32_t split_warps(const QueryArgs& a) {
    if (a.order) return 1;
    const uint64_t sms = sm_count();
    uint32_t wpq = 1;
    const uint64_t entries = std::min(2ull * a.p * a.ix.lists, 1ull * a.ix.rows * a.ix.P.curves);
    const uint64_t worth = a.ix.P.dtype == HC_F32 ? (128u << 10) / a.ix.row_bytes : 1024;
    while (wpq < (uint32_t)kSplitWarps) {
        const uint32_t w = 2 * wpq;
        const bool far = w <= (uint32_t)kSplitBlock && (a.p_query || entries >= w * worth);
        if ((uint64_t)a.nq * w > sms * (w == 2 || far ? 16 : (w == 8 ? 8 : 6))) break;
        wpq = w;
    }
    if (wpq == 2 && !a.p_query && (a.p < 16 || entries < (a.k <= 32 ? 384 : 4096))) return 1;
    return wpq;
}

}  // namespace

cudaError_t launch_query(const IndexView& ix, const void* q, uint32_t nq, uint32_t k, uint32_t p,
                         int32_t* out_ids, void* out_dist, cudaStream_t s,
                         const uint32_t* p_query, const int64_t* pos_in,
                         const uint32_t* order, const uint32_t* pos_cm) {
    if (nq == 0) return cudaSuccess;
    QueryArgs a{ix, q, nq, k, p, out_ids, out_dist, nullptr, p_query, pos_in, order, pos_cm};
    const uint32_t wpq = split_warps(a);
    if (wpq > 1) return launch_split(a, wpq, s);
    const Walk walk = walk_kind(a);
    if (walk == kSweeps) return launch_sweeps(a, s);
    return dispatch<QueryLaunch>(ix.P.dtype == HC_F32, lanes_per_row(ix.row_bytes), regs_for_k(k),
                                 a, walk, s);
}

cudaError_t launch_order_keys(const IndexView& ix, const void* q, uint32_t nq, uint32_t ncurves,
                              uint64_t* keys, uint64_t* qhi, uint64_t* qlo, cudaStream_t s) {
    if (nq == 0 || ncurves == 0) return cudaSuccess;
    order_keys_kernel<<<(unsigned)(((uint64_t)nq + 255) / 256), 256, 0, s>>>(ix, static_cast<const uint8_t*>(q), nq,
                                                       ncurves, keys, qhi, qlo);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_batch_positions(const IndexView& ix, uint32_t nq, const uint32_t* order,
                                   const uint64_t* qhi, const uint64_t* qlo, uint32_t* pos,
                                   cudaStream_t s) {
    const uint32_t qpl = batch_queries_per_lane(ix.lists / ix.P.curves), span = 32 * qpl;
    const uint64_t warps = (((uint64_t)nq + span - 1) / span) * ix.P.curves;
    if (warps == 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((warps + 7) / 8);
    if (qpl == 4)
        batch_positions_kernel<4><<<blocks, 256, 0, s>>>(ix, nq, order, qhi, qlo, pos);
    else if (qpl == 2)
        batch_positions_kernel<2><<<blocks, 256, 0, s>>>(ix, nq, order, qhi, qlo, pos);
    else
        batch_positions_kernel<1><<<blocks, 256, 0, s>>>(ix, nq, order, qhi, qlo, pos);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_fence(const uint64_t* keys_hi, uint64_t total, uint64_t* fence,
                         cudaStream_t s) {
    const uint64_t len = (total + 15) >> kFenceShift;
    if (len == 0) return cudaSuccess;
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint64_t want = (len + 255) / 256, cap = (uint64_t)std::max(sms, 1) * 8;
    fence_kernel<<<(unsigned)std::min(want, cap), 256, 0, s>>>(keys_hi, len, fence);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_positions(const IndexView& ix, const void* q, uint32_t nq, int64_t* pos,
                             cudaStream_t s) {
    if (nq == 0) return cudaSuccess;
    QueryArgs a{ix, q, nq, 1, 0, nullptr, nullptr, pos, nullptr, nullptr, nullptr};
    const unsigned blocks = (unsigned)(((uint64_t)nq + kQWarps - 1) / kQWarps);
    positions_kernel<<<blocks, kQWarps * 32, sizeof(uint32_t) * kQWarps * ix.lists, s>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace hc
