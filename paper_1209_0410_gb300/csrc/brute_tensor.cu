// Exact kNN (Eq. 3) of uint8 rows as a contraction on the tensor cores.
//
// |q - b|^2 = |q|^2 - (2 q.b - |b|^2) with both sides shifted by -128: the
// shifted coordinates are integers of at most 8 bits, exact in float16, and for
// d <= 256 every partial sum of the score 2 q.b - |b|^2 and every distance
// stays below 2^24, so the float32 accumulators hold exact integers and the
// distances equal those of the integer path bit for bit.  2 q is the A operand;
// |b|^2 enters as one more K step, its three base-256 digits against the
// constants -32768 (on twice the digit), -256 and -1.
//
// One block (one per SM) holds MT x 128 queries as the A operand and streams a
// share of the rows as B tiles of NB.  At the end the per-query lists of a
// cluster's blocks meet in distributed shared memory, and each cluster merges its
// lists into the output rows under a lock per row (the row's first id word), so
// nothing is allocated and every SM has a share.  A block in which a wait runs out
// offers no list: its cluster marks its output rows kGaveUp, a mark that no merge
// replaces, and launch_bruteforce searches marked rows again.  Warps:
//   0 .. 4 MT - 1   epilogue, one query per thread (tensor-memory lane): the
//                   scores against the query's threshold; the few that pass are
//                   appended to the query's list in shared memory, which the
//                   warp sorts when it is full
//   4 MT .. + 7     producers: 16-byte loads of the rows, uint8 -> float16 by a
//                   byte permute and one subtraction, stored in 128-byte
//                   swizzled atoms; |b|^2 by dp4a
//   4 MT + 8        one thread issues tcgen05.mma (M 128, N NB, K 16)
// B tiles and accumulators are double-buffered, a group of four producer warps
// per stage.
//
// Bound: the tensor cores' dense float16 rate (5.1 TFLOP for 2,000 queries on
// 10M rows of 128, 2.6 ms at 1940 TFLOP/s).  Measured there: 5.0 ms against 633 ms
// with vabsdiff and dp4a, one warp per query (7.1 with one cluster of 12 blocks
// per query tile, which left 56 SMs idle); one query: 0.63 ms.  A stage waits for
// its refill: one query tile per block, half the tensor work, takes 1,260 cycles
// per row tile where two take 1,850.  Counters (2M rows): tensor pipe 31% busy, shared-
// memory pipe 20%, issue slots 43%, DRAM 2%; the producers wait for their loads.
#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "hc_internal.h"
#include "hc_query_dev.cuh"
#include "hc_tcgen05.cuh"
#include "hc_topk.cuh"

namespace cg = cooperative_groups;

namespace hc {

namespace {

constexpr int kProducers = 8;   // producer warps (4 instead: 13.0 against 9.0 ms)
constexpr int kBBufs = 2;       // B stages and accumulator buffers

// ATOMS: 64-coordinate swizzle atoms per row; KS: list slots per query
// MT: query tiles of 128; NB: rows per B tile (what fits 227 KB with the lists)
template <int ATOMS, int KS, int MT>
struct BruteShape {
    static constexpr int NB = KS == 32 && ATOMS <= 2 ? 128 : 64;
    static constexpr int kQueries = 128 * MT;
    static constexpr int kThreads = 32 * (4 * MT + kProducers + 1);
    static constexpr uint32_t kABytes = (uint32_t)kQueries * ATOMS * 128;
    static constexpr uint32_t kBBytes = (uint32_t)NB * ATOMS * 128;
    static constexpr uint32_t kATail = (uint32_t)kQueries * 32;   // the |b|^2 K step
    static constexpr uint32_t kBTail = (uint32_t)NB * 32;
    static constexpr uint32_t kCols = (uint32_t)(kBBufs * MT * NB);
    static constexpr size_t kSmem = 1024 + kABytes + kATail + kBBufs * (kBBytes + kBTail) +
                                    sizeof(uint64_t) * kQueries * KS + 128;
};

struct BruteArgs {
    const uint8_t* db;
    const uint8_t* q;
    uint64_t n;
    uint32_t row_bytes, nq, k;
    uint32_t groups;   // clusters that share a query tile
    int32_t* out_ids;
    uint32_t* out_dist;
};

constexpr int32_t kLocked = -3;   // no id: ids are >= 0, -1 marks an empty slot

// Looks at a barrier or a row lock before a role gives up.  (The tests build this
// file with 0 and 1, so that waits run out; the wait for tensor-core work in flight
// always has kWaitTries.)
#ifndef HC_BRUTE_TRIES
#define HC_BRUTE_TRIES kWaitTries
#endif
constexpr uint32_t kTries = HC_BRUTE_TRIES;

// empty output rows, which the clusters then merge into
__global__ void __launch_bounds__(256) empty_rows_kernel(uint64_t n, int32_t* ids, uint32_t* dist) {
    const uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    ids[i] = -1;
    dist[i] = 0x7FFFFFFFu;
}

// 16 uint8 coordinates, shifted by -128, as float16 (bytes 0x64 above each
// coordinate make 1024 + x; 1152 is subtracted)
__device__ __forceinline__ void shift_to_half(uint4 v, __half2 (&h)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    const __half2 off = __half2half2(__ushort_as_half(0x6480));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t lo = __byte_perm(w[i], 0x64646464u, 0x4140);
        const uint32_t hi = __byte_perm(w[i], 0x64646464u, 0x4342);
        h[2 * i] = __hsub2(*reinterpret_cast<const __half2*>(&lo), off);
        h[2 * i + 1] = __hsub2(*reinterpret_cast<const __half2*>(&hi), off);
    }
}
// sum of squares of the 16 shifted coordinates
__device__ __forceinline__ int shifted_square(uint4 v) {
    int sq = 0, s;
    s = (int)(v.x ^ 0x80808080u), sq = __dp4a(s, s, sq);
    s = (int)(v.y ^ 0x80808080u), sq = __dp4a(s, s, sq);
    s = (int)(v.z ^ 0x80808080u), sq = __dp4a(s, s, sq);
    s = (int)(v.w ^ 0x80808080u), sq = __dp4a(s, s, sq);
    return sq;
}

// The 32 bytes of vector v (16 coordinates) of row r of a swizzled operand of
// `rows` rows: atom v / 4, 16-byte chunks 2 (v % 4) and the next, each xored
// with the row's low three bits.  Lanes of the upper atom of a pair store
// their chunks in the other order, so that the eight lanes of a row touch
// eight different bank groups.
__device__ __forceinline__ void store_vec(uint8_t* base, uint32_t rows, uint32_t r, uint32_t v,
                                          const __half2 (&h)[8]) {
    const uint4 a = *reinterpret_cast<const uint4*>(&h[0]);
    const uint4 b = *reinterpret_cast<const uint4*>(&h[4]);
    const uint32_t atom = v >> 2, c = 2 * (v & 3), odd = atom & 1;
    uint8_t* p = base + (size_t)atom * rows * 128 + r * 128;
    const uint32_t c0 = (c + odd) ^ (r & 7), c1 = (c + 1 - odd) ^ (r & 7);
    *reinterpret_cast<uint4*>(p + 16 * c0) = odd ? b : a;
    *reinterpret_cast<uint4*>(p + 16 * c1) = odd ? a : b;
}

// three halves (then zeros) as a 16-byte chunk
__device__ __forceinline__ uint4 three_halves(float x, float y, float z) {
    const __half2 a = __floats2half2_rn(x, y), b = __floats2half2_rn(z, 0.f);
    return make_uint4(*reinterpret_cast<const uint32_t*>(&a),
                      *reinterpret_cast<const uint32_t*>(&b), 0u, 0u);
}

// A query's list of KS slots: the best k in order, then `pending` appended
// ones.  The whole warp sorts it; returns the k-th entry.
template <int KS>
__device__ __noinline__ uint64_t sort_list(uint64_t* list, uint32_t k, uint32_t pending,
                                           int lane) {
    constexpr int KR = KS / 32;
    WarpTopK<KR> top;
#pragma unroll
    for (int r = 0; r < KR; ++r) {
        const uint32_t e = r * 32 + lane;
        top.v[r] = e < k + pending ? list[e] : kEmpty;
    }
    sort_all<KR>(top.v, lane);
#pragma unroll
    for (int r = 0; r < KR; ++r) list[r * 32 + lane] = top.v[r];
    __syncwarp();
    return top.kth(k);
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

template <int ATOMS, int KS, int MT>
__global__ void __launch_bounds__(BruteShape<ATOMS, KS, MT>::kThreads, 1)
    brute_tensor_kernel(BruteArgs a) {
    using S = BruteShape<ATOMS, KS, MT>;
    constexpr int NB = S::NB, VP = 4 * ATOMS;   // VP: 16-byte vectors per padded row
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sA = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
    uint8_t* sB = sA + S::kABytes;
    uint8_t* tailA = sB + kBBufs * S::kBBytes;
    uint8_t* tailB = tailA + S::kATail;
    uint64_t* lists = reinterpret_cast<uint64_t*>(tailB + kBBufs * S::kBTail);
    uint64_t* bars = lists + (size_t)S::kQueries * KS;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 4 * kBBufs);
    volatile uint32_t* gave_up = tmem_slot + 1;   // a wait of this block ran out
    const uint32_t bar_full = smem_addr(bars);                 // B stage written
    const uint32_t bar_empty = bar_full + 8 * kBBufs;          // B stage consumed
    const uint32_t bar_done = bar_empty + 8 * kBBufs;          // accumulators complete
    const uint32_t bar_drained = bar_done + 8 * kBBufs;        // accumulators read

    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank(), blocks = cluster.num_blocks();
    const uint32_t shares = blocks * a.groups, share = blockIdx.x % shares;
    const uint32_t q0 = (blockIdx.x / shares) * S::kQueries;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t tiles = (a.n + NB - 1) / NB;
    const uint64_t t0 = tiles * share / shares, t1 = tiles * (share + 1) / shares;
    const uint32_t mytiles = (uint32_t)(t1 - t0);
    const uint32_t vecs = a.row_bytes >> 4;

    // A: twice the block's queries, and the constants of the |b|^2 digits (the
    // upper half of that K step stays zero on both sides); lists empty
    for (uint32_t i = threadIdx.x; i < (uint32_t)(S::kQueries * VP); i += S::kThreads) {
        const uint32_t r = i / VP, v = i % VP;
        __half2 h[8];
        shift_to_half(q0 + r < a.nq && v < vecs
                          ? ldg16(a.q + (size_t)(q0 + r) * a.row_bytes + v * 16)
                          : make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u),
                      h);
#pragma unroll
        for (int j = 0; j < 8; ++j) h[j] = __hadd2(h[j], h[j]);
        store_vec(sA, S::kQueries, r, v, h);
    }
    for (uint32_t i = threadIdx.x; i < S::kATail / 16; i += S::kThreads)
        reinterpret_cast<uint4*>(tailA)[i] = i < (uint32_t)S::kQueries
                                                 ? three_halves(-32768.f, -256.f, -1.f)
                                                 : make_uint4(0, 0, 0, 0);
    for (uint32_t i = threadIdx.x; i < kBBufs * S::kBTail / 16; i += S::kThreads)
        reinterpret_cast<uint4*>(tailB)[i] = make_uint4(0, 0, 0, 0);
    for (uint32_t i = threadIdx.x; i < (uint32_t)(S::kQueries * KS); i += S::kThreads)
        lists[i] = kEmpty;
    if (threadIdx.x == 0) {
        *gave_up = 0;
        for (int i = 0; i < kBBufs; ++i) {
            mbar_init(bar_full + 8 * i, kProducers / kBBufs);
            mbar_init(bar_empty + 8 * i, 1);
            mbar_init(bar_done + 8 * i, 1);
            mbar_init(bar_drained + 8 * i, 4 * MT);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_async_shared();
    if (warp == 4 * MT + kProducers) tmem_alloc(smem_addr(tmem_slot), S::kCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // A role that gives up on a wait says so and ends its loop; the others then run
    // out of their own bounded waits, and the block still reaches the barriers below.
    if (warp < 4 * MT) {
        // ------------------------------------------------ epilogue
        const uint32_t m = warp >> 2, ql = (uint32_t)warp * 32 + lane;   // query of the block
        const uint32_t qi = q0 + ql;
        uint64_t* wl = lists + (size_t)warp * 32 * KS;
        uint64_t* mine = wl + (size_t)lane * KS + a.k;
        int qsq = 0;
        if (qi < a.nq)
            for (uint32_t v = 0; v < vecs; ++v)
                qsq += shifted_square(ldg16(a.q + (size_t)qi * a.row_bytes + v * 16));
        const float qq = (float)qsq;
        // rows whose score reaches thr may enter (distance <= the k-th); the
        // scores of rows past the end are below kNone
        constexpr float kNone = -1.0e9f;
        float thr = qi < a.nq ? kNone : -kNone;
        const uint32_t room = (uint32_t)KS - a.k;
        uint32_t pending = 0;
        auto tidy = [&](uint32_t which) {   // sort the lists of these lanes' queries
            while (which) {
                const int src = __ffs(which) - 1;
                which &= which - 1;
                const uint32_t p = __shfl_sync(0xffffffffu, pending, src);
                const uint64_t kth = sort_list<KS>(wl + (size_t)src * KS, a.k, p, lane);
                if (lane == src) {
                    pending = 0;
                    if (kth != kEmpty) thr = qq - (float)(uint32_t)(kth >> 32);
                }
            }
        };
        // 32 accumulator columns (scores of rows row0 ..) against thr
        auto look_over = [&](const uint32_t (&d)[32], uint32_t at, uint32_t row0) {
            float best[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const uint32_t* x = d + 8 * g;
                best[g] = max3(__uint_as_float(x[0]), __uint_as_float(x[1]),
                               __uint_as_float(x[2]));
                best[g] = max3(best[g], __uint_as_float(x[3]), __uint_as_float(x[4]));
                best[g] = max3(best[g], __uint_as_float(x[5]), __uint_as_float(x[6]));
            }
            const float b0 = max3(best[0], __uint_as_float(d[7]), __uint_as_float(d[15]));
            const float b1 = max3(best[1], __uint_as_float(d[23]), __uint_as_float(d[31]));
            const float top = max3(max3(b0, b1, best[2]), best[3], best[3]);
            if (!__any_sync(0xffffffffu, top >= thr)) return;
            // which columns: then each again, one tensor-memory column at a time
            uint32_t pass = 0;
#pragma unroll
            for (int j = 0; j < 32; ++j) pass |= __uint_as_float(d[j]) >= thr ? 1u << j : 0u;
            uint32_t todo = __reduce_or_sync(0xffffffffu, pass);
            while (todo) {
                const int j = __ffs(todo) - 1;
                todo &= todo - 1;
                const float s = __uint_as_float(tmem_ld1(at + j));
                tmem_ld_wait();
                const uint32_t row = row0 + (uint32_t)j;
                if (s >= thr && row < a.n)
                    mine[pending++] =
                        ((uint64_t)(uint32_t)__float2int_rn(qq - s) << 32) | (uint64_t)row;
                __syncwarp();
                tidy(__ballot_sync(0xffffffffu, pending == room));
            }
        };
        uint32_t i = 0;   // row tile of the share
        for (; i < mytiles; ++i) {
            const uint32_t buf = i % kBBufs, par = (i / kBBufs) & 1;
            if (!mbar_wait_warp(bar_done + 8 * buf, par, kTries)) break;
            tc_fence_after();
            const uint32_t acc = tmem + ((uint32_t)(warp & 3) << 21) + (buf * MT + m) * NB;
            const uint32_t row0 = (uint32_t)(t0 + i) * NB;
            // the next 32 columns are on their way while these are looked over
            uint32_t d[2][32];
            tmem_ld32(acc, d[0]);
#pragma unroll
            for (int c = 0; c < NB / 32; ++c) {
                tmem_ld_wait();
                if (c + 1 < NB / 32) tmem_ld32(acc + 32 * (c + 1), d[(c + 1) & 1]);
                look_over(d[c & 1], acc + 32 * c, row0 + 32 * c);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_drained + 8 * buf);
        }
        if (i < mytiles) *gave_up = 1;
        __syncwarp();
        tidy(__ballot_sync(0xffffffffu, pending > 0));
    } else if (warp < 4 * MT + kProducers) {
        // ------------------------------------------------ producers
        // kBBufs groups of warps, each filling its own stage with every
        // kBBufs-th tile
        constexpr int kPT = kProducers / kBBufs * 32;
        constexpr int kPer = NB * VP / kPT;   // vectors per thread and tile
        static_assert(NB * VP % kPT == 0 && kPer <= VP && kPT / VP % 8 == 0, "whole rounds");
        const uint32_t group = (threadIdx.x - 4 * MT * 32) / kPT;
        const uint32_t pt = (threadIdx.x - 4 * MT * 32) % kPT;
        const uint32_t pr = pt / VP, pv = pt % VP;   // this thread's vector of rows pr + u kPT / VP
        const uint8_t* src = a.db + (size_t)pr * a.row_bytes + pv * 16;
        // a tile's vectors are loaded while the tile before it is converted
        auto load = [&](uint64_t t, uint4 (&x)[kPer]) {
            const uint8_t* p = src + t * NB * a.row_bytes;
            const bool whole = t < t1 && (t + 1) * NB <= a.n && vecs == VP;
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                const uint32_t r = (uint32_t)u * (kPT / VP);
                x[u] = whole || (t < t1 && t * NB + pr + r < a.n && pv < vecs)
                           ? ldg16(p + (size_t)r * a.row_bytes)
                           : make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
            }
        };
        uint4 x[kPer], ahead[kPer];
        load(t0 + group, ahead);
        uint64_t t = t0 + group;
        for (; t < t1; t += kBBufs) {
            const uint32_t i = (uint32_t)(t - t0), buf = i % kBBufs, par = (i / kBBufs) & 1;
            int sq[kPer];
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                x[u] = ahead[u];
                sq[u] = shifted_square(x[u]);
            }
            load(t + kBBufs, ahead);
            // |b|^2: the kPer sums over the row's VP lanes, halving the sums
            // with the lanes; lane v ends with the sum of unit v / (VP / kPer)
            int left = kPer;
#pragma unroll
            for (int o = VP / 2; o >= 1; o >>= 1) {
                if (left > 1) {
                    left /= 2;
                    const bool upper = (pv & (uint32_t)o) != 0;
#pragma unroll
                    for (int u = 0; u < kPer / 2; ++u) {
                        if (u >= left) break;
                        const int send = upper ? sq[u] : sq[u + left];
                        const int keep = upper ? sq[u + left] : sq[u];
                        sq[u] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                } else {
                    sq[0] += __shfl_xor_sync(0xffffffffu, sq[0], o);
                }
            }
            if (!mbar_wait_warp(bar_empty + 8 * buf, par ^ 1, kTries)) break;
            uint8_t* b = sB + buf * S::kBBytes;
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                __half2 h[8];
                shift_to_half(x[u], h);
                store_vec(b, NB, pr + (uint32_t)u * (kPT / VP), pv, h);
            }
            if (pv % (VP / kPer) == 0) {
                const uint32_t r = pr + pv / (VP / kPer) * (kPT / VP);
                const uint32_t n2 = (uint32_t)sq[0];
                *reinterpret_cast<uint4*>(tailB + buf * S::kBTail + r * 16) =
                    t * NB + r < a.n ? three_halves(2.f * (float)(n2 >> 16),
                                                    (float)((n2 >> 8) & 255u), (float)(n2 & 255u))
                                     : three_halves(65504.f, 0.f, 0.f);
            }
            fence_async_shared();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_full + 8 * buf);
        }
        if (t < t1) *gave_up = 1;
    } else if (lane == 0) {
        // ------------------------------------------------ MMA issue
        constexpr uint32_t idesc = mma_idesc_f16(128, NB);
        uint32_t issued = 0;   // row tiles of the share
        for (; issued < mytiles; ++issued) {
            const uint32_t buf = issued % kBBufs, par = (issued / kBBufs) & 1;
            if (!mbar_wait(bar_drained + 8 * buf, par ^ 1, kTries)) break;
            if (!mbar_wait(bar_full + 8 * buf, par, kTries)) break;
            tc_fence_after();
            const uint32_t b = smem_addr(sB) + buf * S::kBBytes;
            const uint64_t bt = mma_desc_plain(smem_addr(tailB) + buf * S::kBTail, NB * 16);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const uint32_t d = tmem + (buf * MT + m) * NB;
#pragma unroll
                for (int s = 0; s < 4 * ATOMS; ++s) {
                    const uint32_t in_atom = (uint32_t)(s % 4) * 32;
                    const uint32_t as = smem_addr(sA) + (uint32_t)(s / 4) * S::kQueries * 128 +
                                        (uint32_t)m * 128 * 128 + in_atom;
                    const uint32_t bs = b + (uint32_t)(s / 4) * NB * 128 + in_atom;
                    mma_f16(d, mma_desc_sw128(as), mma_desc_sw128(bs), idesc, s > 0);
                }
                mma_f16(d, mma_desc_plain(smem_addr(tailA) + m * 128 * 16, S::kQueries * 16), bt,
                        idesc, true);
            }
            mma_commit(bar_empty + 8 * buf);
            mma_commit(bar_done + 8 * buf);
        }
        // the tensor core is done with shared and tensor memory before they go
        bool whole = issued == mytiles;
        for (uint32_t i = issued > kBBufs ? issued - kBBufs : 0; i < issued; ++i)
            whole &= mbar_wait(bar_done + 8 * (i % kBBufs), (i / kBBufs) & 1, kWaitTries);
        if (!whole) *gave_up = 1;
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 4 * MT + kProducers) {
        tc_fence_after();
        tmem_free(tmem, S::kCols);
    }
    // Queries are dealt out to the cluster's blocks: each merges every block's
    // sorted list of its queries (the smaller of entry e of one and entry KS - 1 -
    // e of the other are the KS smallest, a bitonic sequence) and puts the result
    // out.  The clusters of a tile begin at different queries.
    cluster.sync();
    constexpr int KR = KS / 32, kWarps = S::kThreads / 32;
    const uint32_t turn = S::kQueries / blocks / kWarps * (share / blocks) / a.groups;
    const uint32_t rounds = (S::kQueries + blocks * kWarps - 1) / (blocks * kWarps);
    bool whole = true;
    for (uint32_t b = 0; b < blocks; ++b)
        whole &= *cluster.map_shared_rank(tmem_slot + 1, b) == 0;
    for (uint32_t i = 0; i < rounds; ++i) {
        const uint32_t ql = rank + blocks * ((uint32_t)warp + kWarps * ((i + turn) % rounds));
        if (ql >= (uint32_t)S::kQueries || q0 + ql >= a.nq) continue;
        int32_t* ids = a.out_ids + (size_t)(q0 + ql) * a.k;
        uint32_t* dist = a.out_dist + (size_t)(q0 + ql) * a.k;
        if (!whole) {
            if (lane == 0) atomicExch(ids, kGaveUp);
            continue;
        }
        WarpTopK<KR> top;
        top.init();
        for (uint32_t b = 0; b < blocks; ++b) {
            const uint64_t* other = cluster.map_shared_rank(lists + (size_t)ql * KS, b);
#pragma unroll
            for (int r = 0; r < KR; ++r)
                top.v[r] = min(top.v[r], other[KS - 1 - (r * 32 + lane)]);
            merge_sorted<KR>(top.v, lane);
        }
        if (a.groups == 1) {
            top.template store<false>(a.k, lane, ids, dist);
            continue;
        }
        // take the row: its first id word says kLocked meanwhile (a holder lets go in
        // microseconds); a mark found there, or left by giving up, is put back
        int32_t first = kLocked;
        if (lane == 0) {
            for (uint32_t i = 0; i < kTries && first == kLocked; ++i)
                first = atomicExch(ids, kLocked);
            if (first == kLocked || first == kGaveUp) first = kGaveUp, atomicExch(ids, kGaveUp);
        }
        first = __shfl_sync(0xffffffffu, first, 0);
        if (first == kGaveUp) continue;
        __threadfence();
#pragma unroll
        for (int r = 0; r < KR; ++r) {
            const uint32_t e = KS - 1 - (r * 32 + lane);   // reversed, as above
            const int32_t id = e >= a.k ? -1 : (e == 0 ? first : __ldcg(ids + e));
            const uint64_t x =
                id < 0 ? kEmpty : ((uint64_t)__ldcg(dist + e) << 32) | (uint32_t)id;
            top.v[r] = min(top.v[r], x);
        }
        merge_sorted<KR>(top.v, lane);
#pragma unroll
        for (int r = 0; r < KR; ++r) {
            const uint32_t e = r * 32 + lane;
            if (e >= a.k) continue;
            const bool empty = top.v[r] == kEmpty;
            if (e > 0) __stcg(ids + e, empty ? -1 : (int32_t)(uint32_t)top.v[r]);
            __stcg(dist + e, empty ? 0x7FFFFFFFu : (uint32_t)(top.v[r] >> 32));
        }
        __threadfence();
        __syncwarp();
        // let go, unless the row was marked meanwhile
        if (lane == 0)
            atomicCAS(ids, kLocked, top.v[0] == kEmpty ? -1 : (int32_t)(uint32_t)top.v[0]);
    }
    cluster.sync();
}

// How a query tile's rows are shared out: `blocks` per cluster (their lists meet
// in shared memory), `groups` clusters per tile (each merges its lists into the
// output rows, one after the other when they end together: about 3.5 us each).
// A row tile takes a block about 0.65 us, so more than sqrt(btiles / 10.8)
// clusters of two cost more than they save; up to that the chip is filled (`fit`
// clusters of two at once).  (Measured on tiles of 128 rows of 128 bytes, 0.61 us with
// one query tile and 0.89 with two; the time is flat about the best count: at 0.89 us
// that is 17% higher, for 1% of the time.  Other tiles were not measured.)  A few row
// tiles are left to one cluster of eight.
struct Sharing {
    uint32_t blocks, groups;
};
Sharing pick_sharing(uint32_t fit, uint64_t qtiles, uint64_t btiles) {
    if (btiles < 256) {
        uint32_t blocks = 8;
        while (blocks > 1 && btiles < 2 * blocks) blocks /= 2;
        return {blocks, 1};
    }
    const uint64_t chip = std::max<uint64_t>(1, fit / qtiles);
    const uint64_t worth = (uint64_t)std::sqrt((double)btiles / 10.8);
    return {2, (uint32_t)std::min(chip, worth)};
}

template <int ATOMS, int KS, int MT>
cudaError_t launch_tensor(BruteArgs a, cudaStream_t s) {
    using S = BruteShape<ATOMS, KS, MT>;
    auto kernel = brute_tensor_kernel<ATOMS, KS, MT>;
    cudaError_t e = allow_shared(kernel, S::kSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.blockDim = dim3(S::kThreads);
    cfg.dynamicSmemBytes = S::kSmem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    at.val.clusterDim.x = 2;
    cfg.gridDim = dim3(2);
    int fit = 0;
    if ((e = cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg)) != cudaSuccess) return e;
    const uint64_t qtiles = ((uint64_t)a.nq + S::kQueries - 1) / S::kQueries;
    const Sharing sharing =
        pick_sharing((uint32_t)std::max(fit, 1), qtiles, (a.n + S::NB - 1) / S::NB);
    a.groups = sharing.groups;
    at.val.clusterDim.x = sharing.blocks;
    cfg.gridDim = dim3((unsigned)(qtiles * a.groups * sharing.blocks));
    if (a.groups > 1) {
        const uint64_t slots = (uint64_t)a.nq * a.k;
        empty_rows_kernel<<<(unsigned)((slots + 255) / 256), 256, 0, s>>>(slots, a.out_ids,
                                                                         a.out_dist);
        count_launches(1);
    }
    e = cudaLaunchKernelEx(&cfg, kernel, a);
    count_launches(1);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace

// Lists keep at least 16 slots for candidates not yet sorted in (fewer would be
// sorted too often): k <= 16 in 32 slots, then what shared memory holds beside
// the operands, 112 of 128 slots for rows of 128 bytes and 48 of 64 for wider.
bool brute_tensor_takes(uint32_t row_bytes, uint32_t k) {
    return row_bytes <= 256 && k <= (row_bytes <= 128 ? 112u : 48u);
}

cudaError_t launch_brute_tensor(const void* db, uint64_t n, uint32_t row_bytes, const void* q,
                                uint32_t nq, uint32_t k, int32_t* out_ids, void* out_dist,
                                cudaStream_t s) {
    const BruteArgs a{static_cast<const uint8_t*>(db), static_cast<const uint8_t*>(q), n,
                      row_bytes, nq, k, 1, out_ids, static_cast<uint32_t*>(out_dist)};
    // two query tiles per block halve the row conversions
    const bool two = nq > 128;
    if (row_bytes <= 64) {
        if (k > 16) return launch_tensor<1, 128, 1>(a, s);
        return two ? launch_tensor<1, 32, 2>(a, s) : launch_tensor<1, 32, 1>(a, s);
    }
    if (row_bytes <= 128) {
        if (k > 16) return launch_tensor<2, 128, 1>(a, s);
        return two ? launch_tensor<2, 32, 2>(a, s) : launch_tensor<2, 32, 1>(a, s);
    }
    return k > 16 ? launch_tensor<4, 64, 1>(a, s) : launch_tensor<4, 32, 1>(a, s);
}

}  // namespace hc
