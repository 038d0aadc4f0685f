// Exact kNN (Eq. 3) over every row of the database: the ground truth for
// recall, with the same distance and top-k code as the query kernel.  uint8
// batches over enough rows go to brute_tensor.cu.
#include "hc_dispatch.cuh"
#include "hc_internal.h"
#include "hc_query_dev.cuh"
#include "hc_topk.cuh"

namespace hc {

namespace {

constexpr int kQWarps = 8;

// Exact kNN: every row of the database, 32 rows per step, same distance and
// top-k code as the query kernel.  AGAIN: only the queries whose output row the
// kernel before marked kGaveUp (a kernel of its own: with the test at run time the
// search of all queries took 2.5% longer for k <= 32).
template <bool F32, int LPR, int KR, bool AGAIN>
__global__ void __launch_bounds__(kQWarps * 32) brute_kernel(const uint8_t* __restrict__ db,
                                                            uint64_t n, uint32_t row_bytes,
                                                            const uint8_t* __restrict__ q,
                                                            uint32_t nq, uint32_t k,
                                                            int32_t* out_ids, void* out_dist) {
    if constexpr (AGAIN) asm volatile("griddepcontrol.wait;" ::: "memory");   // for the marks
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t qi = blockIdx.x * kQWarps + warp;
    if (qi >= nq || (AGAIN && out_ids[(size_t)qi * k] != kGaveUp)) return;
    const uint8_t* qrow = q + (size_t)qi * row_bytes;
    const uint32_t s = (uint32_t)lane % LPR;
    const uint4 qv0 = s < (row_bytes >> 4) ? ldg16(qrow + s * 16) : make_uint4(0, 0, 0, 0);
    WarpTopK<KR> top;
    top.init();
    for (uint64_t base = 0; base < n; base += 32) {
        const uint32_t cnt = n - base < 32 ? (uint32_t)(n - base) : 32u;
        const uint32_t id = (uint32_t)(base + lane);
        uint64_t cand[ChunkWidth<LPR>::NG];
        chunk_candidates_n<F32, LPR>(db, row_bytes, qrow, qv0, id, cnt, lane, cand);
#pragma unroll
        for (int c = 0; c < ChunkWidth<LPR>::NG; ++c) top.offer(cand[c], k, lane);
    }
    top.template store<F32>(k, lane, out_ids + (size_t)qi * k,
                            static_cast<uint32_t*>(out_dist) + (size_t)qi * k);
}

template <bool F32, int LPR, int KR>
struct BruteLaunch {
    static cudaError_t run(const uint8_t* db, uint64_t n, uint32_t row_bytes, const uint8_t* q,
                           uint32_t nq, uint32_t k, int32_t* ids, void* dist, bool again,
                           cudaStream_t s) {
        const unsigned blocks = (nq + kQWarps - 1) / kQWarps;
        if (!again) {
            brute_kernel<F32, LPR, KR, false><<<blocks, kQWarps * 32, 0, s>>>(db, n, row_bytes, q,
                                                                              nq, k, ids, dist);
            count_launches(1);
            return cudaGetLastError();
        }
        if constexpr (F32 || LPR > 16) {
            return cudaErrorInvalidValue;   // brute_tensor_takes: uint8 rows of at most 256 bytes
        } else {
            // starts as the tensor-core kernel ends (2 us a call)
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute at{};
            at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at.val.programmaticStreamSerializationAllowed = 1;
            cfg.gridDim = dim3(blocks);
            cfg.blockDim = dim3(kQWarps * 32);
            cfg.stream = s;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            const cudaError_t e = cudaLaunchKernelEx(&cfg, brute_kernel<F32, LPR, KR, true>, db, n,
                                                     row_bytes, q, nq, k, ids, dist);
            count_launches(1);
            return e == cudaSuccess ? cudaGetLastError() : e;
        }
    }
};

// Rows from which uint8 rows go to the tensor cores.  Below, every query still
// meets many rows that enter its list, and there one warp per query (here)
// beats one warp for 32 queries (there); from there on the time here grows with
// the rows and there with their logarithm.  The line is lower where a row costs
// more here, and higher where a list of 32 or 128 slots leaves less room for
// rows not yet sorted in.  Times here / there, the lower of clustered and uniform
// rows and of 33, 129 and 2,000 queries:
//   rows <= 64 bytes   k = 1: 0.96 at 6,000 rows, 1.12 at 8,192; k = 5: 0.99 at 10,000, 1.13 at
//                      12,288; k = 10: 0.60 at 4,096, 1.00 at 14,000; k = 16: 0.50 at 4,096,
//                      0.99 at 20,000; k = 100: 0.74 at 32,768, 0.91 at 49,152, 1.07 at
//                      65,536; k = 112: 0.51 at 32,768, 0.96 at 98,304, 1.17 at 131,072
//   up to 128 bytes    k <= 10: 1.1 and more at 4,096; k = 16: 0.86 at 4,096, 1.03 at 6,000;
//                      k = 112: 0.81 at 32,768, 1.02 at 49,152
constexpr uint64_t tensor_min_rows(uint32_t row_bytes, uint32_t k) {
    if (k <= 16) {
        if (row_bytes <= 64) return 5500 + 950 * k;
        return row_bytes <= 128 && k > 10 ? 6000 : 4096;
    }
    if (row_bytes > 128) return 32768;
    // k <= 112 (brute_tensor_takes)
    const uint64_t room = k < 128 ? 128 - k : 1, line = (row_bytes <= 64 ? 1650000 : 760000) / room;
    return line > 32768 ? line : 32768;
}

}  // namespace

cudaError_t launch_bruteforce(const void* db, hc_dtype dtype, uint64_t n, uint32_t d,
                              const void* q, uint32_t nq, uint32_t k, int32_t* out_ids,
                              void* out_dist, cudaStream_t s) {
    if (nq == 0) return cudaSuccess;
    const uint32_t row_bytes = dtype == HC_F32 ? d * 4 : d;
    const bool tensor = dtype == HC_U8 && n >= tensor_min_rows(row_bytes, k) &&
                        brute_tensor_takes(row_bytes, k);
    if (tensor) {
        const cudaError_t e = launch_brute_tensor(db, n, row_bytes, q, nq, k, out_ids, out_dist, s);
        if (e != cudaSuccess) return e;
    }
    // all queries, or those the tensor cores gave up
    return dispatch<BruteLaunch>(dtype == HC_F32, lanes_per_row(row_bytes), regs_for_k(k),
                                 static_cast<const uint8_t*>(db), n, row_bytes,
                                 static_cast<const uint8_t*>(q), nq, k, out_ids, out_dist, tensor,
                                 s);
}

}  // namespace hc
