// Internal structures shared by the host runtime (rrs_api.cu) and the kernel
// translation units.  Not part of the public ABI.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/rrs.h"

namespace rrs {

// A resident dataset, as the kernels see it.
struct DsDev {
    const float* X32;      // n x ldx FP32 rows, zero padded
    // Xt: the FP32 data again as columns, for the selection kernels (d <= 16), or nullptr: dim l of point i at
    // l * roundup32(n) + i, zero beyond n, so that a warp's lanes read consecutive points side by side.
    const float* Xt;
    const double* X64;     // n x d FP64 rows, or nullptr if the data came in FP32
    const float* xnorm;    // n Euclidean row norms, rounded up
    const uint16_t* Xbf;   // n x (2*kp) BF16 planes [x_hi | x_lo] for the tensor-core path, or nullptr
    const float* center;   // d: mean of the rows
    const float* cov;      // d x d covariance of the rows (d <= RRS_COV_MAX_D), else nullptr
    int64_t n;
    int32_t d;
    int32_t ldx;           // padded FP32 row stride (floats)
    int32_t kp;            // padded K of one BF16 plane (multiple of 64), 0 if no planes
    float rc;              // max_i |x_i - center| (rounded up): every |u'(x_i - center)| <= rc for |u| <= 1
};

constexpr int RRS_COV_MAX_D = 128;

// One query of a launch (any request, any dataset).
struct SlotDev {
    int32_t ds;            // index into the DsDev array
    int32_t kind;
    int32_t m;             // directions per round
    int32_t r;             // rounds
    float alpha;
    int32_t d;
    int32_t ldx;
    int32_t zdtype;        // 0 = FP32, 1 = FP64
    uint64_t seed;
    int64_t qctr;          // query counter index in the direction stream
    int64_t uoff;          // offset of this slot's m x ldx directions in U (floats)
    int64_t roff;          // offset of this slot's m results / y_z values
    int64_t zoff32;        // offset of the FP32 query row (ldx floats) and of the poles
    int64_t zoff64;        // offset of the FP64 query row (d doubles)
    const void* zsrc;      // caller's query row (device)
    double* depth_out;     // this query's output cells (device), may be null
    int64_t* count_out;
    int32_t* best_out;
    int32_t* choice_out;   // r cells
    // running state (Alg. 1 step 5)
    double dmin;
    int64_t cmin;
    int32_t best;
    float znorm;
    int32_t round;         // next round (0-based) when launched in per-slot round mode
    int32_t pad2;
};

// A block of directions of one slot handled by one CTA.
struct TaskDev {
    int32_t slot;
    int32_t j0;
    int32_t nj;
    int32_t ds;            // selection tasks: the slot's dataset row (read beside the slot, not after it); else 0
};

// Per (slot, direction) result of one round.
struct ResDev {
    double depth;
    int64_t count;         // halfspace: min(#<=, #>=); else -1
};

// Device-side error bits (ORed into one word).
enum : int {
    ERR_SELECT_ITER = 1,    // bucket selection did not converge
    ERR_SELECT_CAP = 2,
    ERR_EXPANSION = 4,      // exact-sign expansion overflow
    ERR_TIMEOUT = 8,
    ERR_TC_SETUP = 16,
};

// Near-tie band factors: a point is re-checked exactly when
// |t| <= gamma * (|x| + |z|), t the fast projection difference.
// FP32 path: |fl32 dot - exact| <= gamma_d sum|u x| (gamma_d ~ d 2^-24), plus one rounding of x to FP32
// (FP64 inputs) and of y_z, from which the chain starts, to FP32; twice that sum for slack.
__host__ __device__ inline float band_gamma_fp32(int d) { return (float)((double)(d + 4) * 0x1p-23); }
float band_gamma_tc(int kp);
// cuTensorMapEncodeTiled, looked up once through the runtime (NULL when unavailable)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_fn();
__host__ __device__ float band_coef_ff(int d);   // bound coefficient of the compensated FP32 re-check (tensor-core path)

// Dynamic shared memory a kernel may ask for: raised once per device to the most its static memory leaves, by the first
// launch there.  The limit belongs to the kernel, not to a launch: one that set its own size on every call could lower
// it between another host thread's setting and that thread's launch.  One object per kernel.
class SmemLimit {
    std::atomic<uint64_t> done_{0};   // devices 0 .. 63 whose limit is raised

public:
    template <class K>
    cudaError_t raise(K* kernel)
    {
        int dev = 0, most = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess && dev < 64 && (done_.load(std::memory_order_acquire) >> dev & 1)) return e;
        cudaFuncAttributes a{};
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, kernel);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes);
        if (e != cudaSuccess)
            cudaGetLastError();   // do not leave the failure pending for an unrelated later call
        else if (dev < 64)
            done_.fetch_or(1ull << dev, std::memory_order_release);
        return e;
    }
};

// Set the text that rrs_last_error() returns on this thread (rrs_api.cu).
void set_last_error(const char* msg);

// launchers (rrs_kernels.cu)
cudaError_t launch_prep(const SlotDev* slots, int nslots, const DsDev* ds, float* z32, double* z64,
                        float* poles, cudaStream_t st);
// max_ldx: the largest row stride among the tasks' queries (sizes the shared-memory staging); res: the result cells
// of the tasks' directions, which are zeroed
cudaError_t launch_gen(const TaskDev* tasks, int ntasks, const SlotDev* slots, const float* poles_cur,
                       const double* z64, float* U, double* yz, ResDev* res, int round0, int max_ldx, cudaStream_t st);
// FP32 halfspace tasks hold up to HD_ROWS consecutive (query, direction) rows; where a request's queries lie in
// consecutive slots they may run from one query into the next (j0 counts within the task's first query)
// split_n: the largest n among the tasks' datasets, which lets a launch of few tasks split the points over more
// CTAs (the result cells must then be zero, as launch_gen leaves them); 0: no split
// max_ldx: the largest row stride among the tasks' datasets (sizes the shared memory), at most HD_MAX_LDX in a call;
// wider rows are refused
constexpr int HD_ROWS = 64;
constexpr int HD_MAX_LDX = 440;
constexpr int HD_PART_SHIFT = 48;   // bits of a count in a result cell shared by the parts of a split (n < 2^48)
cudaError_t launch_hd_simt(const TaskDev* tasks, int ntasks, int max_ldx, int64_t split_n, const SlotDev* slots, const DsDev* ds,
                           const float* U, const double* yz, const double* z64, ResDev* res, int64_t* band_out,
                           int* err, cudaStream_t st);
// group: directions per task and variant: the kernel, both from pdap_shape and shared by every task.  Where a
// request's queries lie in consecutive slots a task may run from one query into the next, as for halfspace.
// yz: the FP64 y_z = u'z of every direction (the direction generator's output), used for the depth.
// Launches the selection kernel, which writes the points holding the order statistics into the result cells,
// then k_pdap_finish, which forms the depths from FP64 projections of those points: PDAP_LAUNCH_KERNELS kernels.
constexpr int PDAP_LAUNCH_KERNELS = 2;
// its selection kernel for the variants PDAP_WARP and PDAP_KEYS (pdap_select.cu)
cudaError_t launch_sel(const TaskDev* tasks, int ntasks, int group, int variant, const SlotDev* slots, const DsDev* ds,
                       const float* U, ResDev* res, int* err, cudaStream_t st, const float* kin);
cudaError_t launch_pdap(const TaskDev* tasks, int ntasks, size_t smem, int group, int variant, const SlotDev* slots,
                        const DsDev* ds, const float* U, const double* yz, ResDev* res, int* err, cudaStream_t st,
                        const float* kin = nullptr);
// Keys of ntasks selection tasks (all of one dataset) into keys (pdap_keys_bytes), for
// launch_pdap(..., kin = keys) on the same task range, with the selection kernel's own key arithmetic:
// a tiled FP32 GEMM for d > 16 (where forming the keys inside the selection kernel re-reads X for every
// G directions), two half chains per key for d <= 16 (where keys in device memory are asked for)
size_t pdap_keys_bytes(int n, int group, int ntasks);
// Bytes of selection keys formed at a time (one chunk of tasks: a keys launch, then the selection on them).  A chunk's
// launches end in waves that are partly empty, so chunks are large: n = 100,000 at d = 100 took 117 / 89 / 74 / 66 ms
// with 64 / 128 / 256 / 512 MB.  Where the context's budget has no room for KEYS_SCRATCH_BYTES the plan takes
// KEYS_SCRATCH_MIN; so does a captured graph, which keeps its workspace, under a budget or where the context's graphs
// hold rrs_ctx::GRAPH_KEEP (32 datasets of up to 50,000 points: 38.3 ms a call with large chunks, 39.1 with small ones).
constexpr size_t KEYS_SCRATCH_BYTES = (size_t)1 << 30, KEYS_SCRATCH_MIN = (size_t)256 << 20;
// Tasks of one keys launch: at most `bytes` of keys and what its grid holds, one at least.
int pdap_keys_chunk(int n, int d, int group, int64_t ntasks, size_t bytes);
cudaError_t launch_pdap_keys(const TaskDev* tasks, int ntasks, int group, const SlotDev* slots, const DsDev* ds,
                             const DsDev& ds_host, const float* U, float* keys, cudaStream_t st);
int pdap_dp4_class(int d);
cudaError_t launch_argmin(SlotDev* slots, const int32_t* slot_list, int nlist, const float* U,
                          const ResDev* res, const float* poles_cur, float* poles_next, int round0,
                          int last_round, cudaStream_t st);
// launch_argmin of round round0 and launch_gen of the next in one launch, for slots of at most NEXT_MAX_M directions
constexpr int NEXT_MAX_M = 128;
cudaError_t launch_next(SlotDev* slots, const int32_t* slot_list, int nlist, const float* poles_cur, float* poles_next,
                        const double* z64, float* U, double* yz, ResDev* res, int round0, int max_ldx, cudaStream_t st);
cudaError_t launch_yz_only(const TaskDev* tasks, int ntasks, const SlotDev* slots, const double* z64,
                           const float* U, double* yz, cudaStream_t st);
cudaError_t launch_scatter_dirs(const SlotDev* slots, int nslots, int m, int d, const float* Uin, float* U,
                                cudaStream_t st);
// Per-slot round mode (serving): each slot runs its own next round S.round; poles0 holds the
// pole of slots at even rounds, poles1 of odd ones; argmin advances S.round.
cudaError_t launch_gen_slotround(const TaskDev* tasks, int ntasks, const SlotDev* slots, const float* poles0,
                                 const float* poles1, const double* z64, float* U, double* yz, ResDev* res,
                                 int max_ldx, cudaStream_t st);
cudaError_t launch_argmin_slotround(SlotDev* slots, const int32_t* slot_list, int nlist, const float* U,
                                   const ResDev* res, float* poles0, float* poles1, cudaStream_t st);
cudaError_t launch_debug_dirs(uint64_t seed, int q, int round0, int m, int d, float alpha, const float* pole,
                              float* U, cudaStream_t st);
cudaError_t launch_convert_dataset(const void* X, int dtype, int64_t n, int d, int ldx, float* X32,
                                   double* X64, float* xnorm, int* bad, cudaStream_t st);
// DsDev::Xt from the padded rows X32 (Xt holds columns_floats(n, d) floats)
size_t columns_floats(int64_t n, int d);
cudaError_t launch_columns(const float* X32, int64_t n, int d, int ldx, float* Xt, cudaStream_t st);
// mean, covariance (d <= RRS_COV_MAX_D) and radius about the mean of the FP32 rows; rc_out is a device float
cudaError_t launch_moments(const float* X32, int64_t n, int d, int ldx, float* center, float* cov, float* rc_out,
                           cudaStream_t st);
cudaError_t launch_check_finite(const void* Z, int dtype, int64_t count, int* bad, cudaStream_t st);
size_t pdap_smem_bytes(int n, int group, int ldx, bool stream = false);
size_t pdap_smem_limit();
// directions per CTA of the allocation-free call for d > 16, 0 where none fits with its keys
int pdap_max_group(int n, int ldx, int m);

// Selection-kernel variant bit: no keys in shared memory, every pass recomputes them from X (the allocation-free
// entry point with d > 16 where they do not fit).  Such launches take PDAP_STREAM_GROUP directions per CTA.
constexpr int PDAP_STREAM = 0x100;
// Largest n the selection kernels take: point indices and the padded key count (n rounded up to 4) are int.
constexpr int64_t PDAP_MAX_N = 0x7FFFFFC0;
constexpr int PDAP_STREAM_GROUP = 2;
// Selection-kernel variant bit: one warp per direction, keys re-formed from X at both passes (d <= 16); the low
// byte holds d, bits 16 up the logarithm of the bucket count.  The default for d <= 16.
constexpr int PDAP_WARP = 0x200;
constexpr int PDAP_WARP_GROUP = RRS_SELECT_WARP;
// Selection-kernel variant bit: keys formed once in device memory (launch_pdap_keys) and read at both passes, one
// block per direction; bits 16 up hold the logarithm of the bucket count.  The default for d > 16.
constexpr int PDAP_KEYS = 0x400;
constexpr int PDAP_KEYS_GROUP = 8;
// pdap_shape group asking for it
constexpr int PDAP_STREAM_CHOICE = RRS_SELECT_STREAM;
inline bool pdap_x_eligible(int d) { return d >= 1 && d <= 16; }
struct PdapShape {
    int group;        // directions per CTA
    int variant;      // pdap_dp4_class(d); or PDAP_WARP | d | log2 nb << 16; or PDAP_KEYS | log2 nb << 16
    size_t smem;      // dynamic shared memory per CTA
    bool keys_gemm;   // keys formed first by launch_pdap_keys
};
// Launch shape for a dataset (n rows, d dims, row stride ldx) and m directions per query.  group: 0 for the default,
// 1, 2 or 4 for that many directions per CTA with resident keys (taken when they fit), PDAP_WARP_GROUP or
// PDAP_STREAM_CHOICE.  rows: (query, direction) rows of the launch, 0 when unknown.
PdapShape pdap_shape(int n, int ldx, int m, int d, int group = 0, int64_t rows = 0);

// tensor-core path (hd_tc.cu)
cudaError_t launch_build_bf16_planes(const float* X32, int64_t n, int d, int ldx, int kp, uint16_t* Xbf,
                                     cudaStream_t st);
// Points per tile of the tensor-core kernel for planes of K extent kp: want = 128 or 256 where both exist
// (kp = 64), anything else for the default.
int tc_tile_n(int kp, int want = 0);
// The tensor map of a dataset's BF16 planes (kp 64 or 128; planes built) for tiles of bn points, written to *out
// (host memory; the caller copies it into the device array passed as maps).
cudaError_t encode_tc_map(const DsDev& ds_host, int bn, CUtensorMap* out);
// tasks of up to 128 (query, direction) rows each, of any datasets whose planes have K extent kp and whose maps
// were encoded for tiles of bn points; maps[ds] is the tensor map of dataset row ds of ds_dev (device memory,
// 64-byte aligned)
// split_n: as for launch_hd_simt
cudaError_t launch_hd_tc(const TaskDev* tasks, int ntasks, int kp, int bn, int64_t split_n, const SlotDev* slots,
                         const DsDev* ds_dev, const CUtensorMap* maps, const float* U, const double* yz,
                         const double* z64, ResDev* res, int64_t* band_out, int* err, cudaStream_t st);
bool hd_tc_supported(int d);
cudaError_t launch_wait_probe(int* err, long long limit_cycles, cudaStream_t st);

}  // namespace rrs
