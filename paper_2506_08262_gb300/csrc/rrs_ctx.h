// Host-side state of a context (shared by the runtime and the serving loop).
// Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "../../include/rrs.h"
#include "rrs_internal.h"

namespace rrs {

struct Dataset {
    int64_t n = 0;
    int32_t d = 0;
    int32_t ldx = 0;
    int32_t kp = 0;
    float* X32 = nullptr;
    float* Xt = nullptr;       // d <= 16: the FP32 data as columns (DsDev::Xt)
    double* X64 = nullptr;
    float* xnorm = nullptr;
    uint16_t* Xbf = nullptr;
    float* center = nullptr;   // d, then (d <= RRS_COV_MAX_D) d*d covariance, then the radius
    float* cov = nullptr;
    float rc = 0.0f;
    size_t bytes = 0;
};

}  // namespace rrs

struct rrs_ctx {
    int device = 0;
    uint64_t budget = 0;
    uint64_t used = 0;
    int64_t next_id = 1;
    std::map<int64_t, rrs::Dataset> datasets;
    uint64_t launches = 0;
    int* d_err = nullptr;
    // pool of the per-call workspaces: the context's own, so that memory stays mapped from one call to the next (the
    // device's default pool gives it back at every synchronisation, and mapping it again costs more than a short
    // call), up to POOL_KEEP bytes; a context with a budget keeps nothing.  Given back by rrs_destroy.
    static constexpr uint64_t POOL_KEEP = (uint64_t)2 << 30;
    cudaMemPool_t pool = nullptr;
    // workspace bytes of cached graphs up to which a further one takes large keys chunks
    static constexpr uint64_t GRAPH_KEEP = (uint64_t)2 << 30;
    int* h_flag = nullptr;   // pinned: device-side flags read back without a staged copy
    std::mutex mu;
    // cached captured graphs of batched calls (keyed by the request bytes)
    struct GraphEntry {
        std::vector<char> key;
        cudaGraphExec_t exec = nullptr;
        void* ws = nullptr;
        size_t ws_bytes = 0;
        size_t launches = 0;
    };
    std::vector<GraphEntry> graphs;
    // selection-kernel autotuning: (n, ldx, m) -> directions per CTA
    std::map<std::tuple<int64_t, int, int>, int> pd_tune;
    std::map<std::pair<int64_t, int>, int> tc_tune;   // (n, kp) -> points per tensor-core tile
    // per-stage CUDA-event timing (rrs_profile_*)
    bool profiling = false;
    struct Mark {
        int stage;
        cudaEvent_t a, b;
    };
    std::vector<Mark> marks;
    std::vector<cudaEvent_t> event_pool;
    double stage_ms[RRS_NSTAGES] = {};
    int64_t stage_launches[RRS_NSTAGES] = {};
};

namespace rrs {
// cudaMalloc for what a context keeps; where memory is short, what its pool holds between calls goes back first.
template <class T>
cudaError_t ctx_malloc(rrs_ctx* ctx, T** p, size_t bytes)
{
    cudaError_t e = cudaMalloc((void**)p, bytes);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    cudaMemPoolTrimTo(ctx->pool, 0);
    return cudaMalloc((void**)p, bytes);
}

// Build (once) the BF16 hi/lo planes the tensor-core halfspace kernel streams;
// UNSUPPORTED for d + 2 > 128, BUDGET when they do not fit the context's budget.
rrs_status ensure_bf16_planes(rrs_ctx* ctx, Dataset& D);
}  // namespace rrs
