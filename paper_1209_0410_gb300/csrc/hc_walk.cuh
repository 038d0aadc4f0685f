// Arguments and shared-memory layout of the walk kernels: one query per warp
// (query.cu), a query per several warps (query_split.cu), rows in sweeps of
// ascending ids (query_sweep.cu).
#pragma once

#include "hc_dispatch.cuh"
#include "hc_internal.h"
#include "hc_query_dev.cuh"
#include "hc_topk.cuh"

namespace hc {

constexpr int kQWarps = 8;       // warps per block, a query each
constexpr int kSplitWarps = 16;  // warps that may share a query
constexpr int kSplitBlock = 8;   // warps per block that share queries (16 for one query)

struct QueryArgs {
    IndexView ix;
    const void* q;
    uint32_t nq, k, p;
    int32_t* out_ids;
    void* out_dist;
    int64_t* out_pos;            // positions-only kernel
    const uint32_t* p_query;     // per-query depth (overrides p), or null
    const int64_t* pos_in;       // precomputed lower_bound positions (nq x lists), or null
    const uint32_t* order;       // warp w answers query order[w], or null (w itself)
    const uint32_t* pos_cm;      // positions of the batch pass (curve-major rows), or null
};

// shared bytes of one warp's row ring
template <int LPR>
__host__ __device__ __forceinline__ uint32_t ring_bytes(uint32_t row_bytes) {
    return LPR <= 8 ? kRingRows * row_bytes : kWideRing;
}

// uint8 rows of at most 128 bytes; order and pos_cm set
cudaError_t launch_sweeps(const QueryArgs& a, cudaStream_t s);
// wpq (a power of two up to kSplitWarps) warps per query; no order
cudaError_t launch_split(const QueryArgs& a, uint32_t wpq, cudaStream_t s);

}  // namespace hc
