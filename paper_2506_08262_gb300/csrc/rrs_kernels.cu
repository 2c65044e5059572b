// RRS round kernels for sm_103a: direction generation (Alg. S1/S4), halfspace
// counts on the CUDA cores with an exact near-tie recheck (Sec. 2, D_H), and
// the round minimum with the pole update (Alg. 1 steps 4-6).  The D_P / D_AP
// selection kernel lives in pdap.cu.
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "packed_fma.cuh"
#include "rrs_device.cuh"
#include "rrs_internal.h"

namespace rrs {

using namespace rrsdev;


// ---------------------------------------------------------------------------
// dataset and query preparation
// ---------------------------------------------------------------------------

template <typename T>
__global__ void k_convert_dataset(const T* __restrict__ X, int64_t n, int d, int ldx, float* __restrict__ X32,
                                  double* __restrict__ X64, float* __restrict__ xnorm, int* bad)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const T* row = X + i * d;
    double s = 0.0;
    int isbad = 0;
    for (int l = 0; l < ldx; ++l) {
        if (l < d) {
            const double v = (double)row[l];
            if (!(fabs(v) < 1.8446744073709552e19)) isbad = 1;  // non-finite or |v| >= 2^64
            s = __fma_rn(v, v, s);
            X32[i * ldx + l] = (float)v;
            if (X64) X64[i * d + l] = v;
        } else {
            X32[i * ldx + l] = 0.0f;
        }
    }
    xnorm[i] = __double2float_ru(__dsqrt_ru(s) * (1.0 + 1e-12));
    if (isbad) atomicOr(bad, 1);
}

cudaError_t launch_convert_dataset(const void* X, int dtype, int64_t n, int d, int ldx, float* X32, double* X64,
                                   float* xnorm, int* bad, cudaStream_t st)
{
    const int nt = 128;
    const int64_t nb = (n + nt - 1) / nt;
    if (dtype == 0)
        k_convert_dataset<float><<<(unsigned)nb, nt, 0, st>>>((const float*)X, n, d, ldx, X32, X64, xnorm, bad);
    else
        k_convert_dataset<double><<<(unsigned)nb, nt, 0, st>>>((const double*)X, n, d, ldx, X32, X64, xnorm, bad);
    return cudaGetLastError();
}

// One thread per (dim, point) of the columns, points beyond n zero.
__global__ void k_columns(const float* __restrict__ X32, int64_t n, int ldx, int64_t colst, float* __restrict__ Xt)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= colst) return;
    const int l = blockIdx.y;
    Xt[l * colst + i] = i < n ? X32[i * ldx + l] : 0.0f;
}

size_t columns_floats(int64_t n, int d) { return (size_t)((n + 31) / 32) * 32 * (size_t)d; }

cudaError_t launch_columns(const float* X32, int64_t n, int d, int ldx, float* Xt, cudaStream_t st)
{
    const int64_t colst = (n + 31) / 32 * 32;
    const int nt = 256;
    const dim3 grid((unsigned)((colst + nt - 1) / nt), (unsigned)d);
    k_columns<<<grid, nt, 0, st>>>(X32, n, ldx, colst, Xt);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// data moments (range heuristics of the selection kernel only; no result
// depends on their accuracy)
// ---------------------------------------------------------------------------

__global__ void k_center(const float* __restrict__ X32, int64_t n, int ldx, float* __restrict__ center)
{
    const int a = blockIdx.x;
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += (double)X32[i * ldx + a];
    __shared__ double red[256];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) center[a] = (float)(red[0] / (double)n);
}

__global__ void k_cov(const float* __restrict__ X32, int64_t n, int d, int ldx, const float* __restrict__ center,
                      float* __restrict__ cov)
{
    const int a = blockIdx.x / d, b = blockIdx.x % d;
    if (b < a) return;
    const float ca = center[a], cb = center[b];
    float s = 0.0f;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s = fmaf(X32[i * ldx + a] - ca, X32[i * ldx + b] - cb, s);
    __shared__ float red[256];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const float v = red[0] / (float)n;
        cov[a * d + b] = v;
        cov[b * d + a] = v;
    }
}

__global__ void k_radius(const float* __restrict__ X32, int64_t n, int d, int ldx, const float* __restrict__ center,
                         float* rc)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
    for (int l = 0; l < d; ++l) {
        const double v = (double)X32[i * ldx + l] - (double)center[l];
        s = __fma_rn(v, v, s);
    }
    const float r = __double2float_ru(__dsqrt_ru(s) * (1.0 + 1e-9));
    atomicMax((int*)rc, __float_as_int(r));   // non-negative floats order like their bit patterns
}

cudaError_t launch_moments(const float* X32, int64_t n, int d, int ldx, float* center, float* cov, float* rc_out,
                           cudaStream_t st)
{
    k_center<<<d, 256, 0, st>>>(X32, n, ldx, center);
    if (cov) k_cov<<<d * d, 256, 0, st>>>(X32, n, d, ldx, center, cov);
    cudaError_t e = cudaMemsetAsync(rc_out, 0, sizeof(float), st);
    if (e != cudaSuccess) return e;
    k_radius<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(X32, n, d, ldx, center, rc_out);
    return cudaGetLastError();
}

template <typename T>
__global__ void k_check_finite(const T* __restrict__ Z, int64_t count, int* bad)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        if (!(fabs((double)Z[i]) < 1.8446744073709552e19)) atomicOr(bad, 1);
}

cudaError_t launch_check_finite(const void* Z, int dtype, int64_t count, int* bad, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    const int nt = 256;
    int64_t nb = (count + nt - 1) / nt;
    if (nb > 4096) nb = 4096;
    if (dtype == 0) k_check_finite<float><<<(unsigned)nb, nt, 0, st>>>((const float*)Z, count, bad);
    else k_check_finite<double><<<(unsigned)nb, nt, 0, st>>>((const double*)Z, count, bad);
    return cudaGetLastError();
}

__global__ void k_prep(SlotDev* slots, int nslots, const DsDev* ds, float* z32, double* z64, float* poles)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nslots) return;
    SlotDev& S = slots[s];
    const int d = S.d, ldx = S.ldx;
    double acc = 0.0;
    for (int l = 0; l < ldx; ++l) {
        double v = 0.0;
        if (l < d) {
            v = S.zdtype == 0 ? (double)((const float*)S.zsrc)[l] : ((const double*)S.zsrc)[l];
            z64[S.zoff64 + l] = v;
            acc = __fma_rn(v, v, acc);
        }
        z32[S.zoff32 + l] = (float)v;
        poles[S.zoff32 + l] = (l == 0) ? 1.0f : 0.0f;
    }
    S.znorm = __double2float_ru(__dsqrt_ru(acc) * (1.0 + 1e-12));
    S.dmin = 1.0;
    S.cmin = ds[S.ds].n;
    S.best = -1;
}

cudaError_t launch_prep(const SlotDev* slots, int nslots, const DsDev* ds, float* z32, double* z64, float* poles,
                        cudaStream_t st)
{
    if (nslots <= 0) return cudaSuccess;
    const int nt = 128;
    k_prep<<<(nslots + nt - 1) / nt, nt, 0, st>>>((SlotDev*)slots, nslots, ds, z32, z64, poles);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// direction generation: one thread per (slot, direction)
// ---------------------------------------------------------------------------

// One thread per direction of one query (a task never spans queries).  With d <= stage_d the CTA builds
// its directions in shared memory, transposed (element i of thread t at i * GEN_STRIDE + t: the passes
// of the generator, the same arithmetic in the same order, touch consecutive banks), and then writes
// the rows out whole, coalesced; larger d builds each row in place in U.
constexpr int GEN_NT = 128, GEN_STRIDE = GEN_NT + 1;
constexpr size_t GEN_STAGE_MAX = 96 * 1024;

// The directions j0 .. j0 + nj - 1 of one query for round rnd around its pole, by a CTA of GEN_NT threads.
__device__ __forceinline__ void gen_rows(const SlotDev& S, int j0, int nj, int rnd, const float* pole,
                                         const double* __restrict__ z64, float* __restrict__ U,
                                         double* __restrict__ yz, ResDev* __restrict__ res, int stage_d, float* gstage)
{
    const int jl = threadIdx.x, j = j0 + jl;
    const float ap = alpha_power(S.alpha, rnd);
    const double* z = z64 + S.zoff64;
    // zero result cells: where the halfspace kernels split the points they add their counts there
    if (jl < nj) res[S.roff + j] = ResDev{0.0, 0};
    if (S.d > stage_d) {
        if (jl >= nj) return;
        float* u = U + S.uoff + (int64_t)j * S.ldx;
        stream_direction(S.seed, (uint32_t)S.qctr, (uint32_t)rnd, (uint32_t)j, S.d, ap, pole, u, 1);
        for (int l = S.d; l < S.ldx; ++l) u[l] = 0.0f;
        double acc = 0.0;
        for (int l = 0; l < S.d; ++l) acc = __fma_rn((double)u[l], z[l], acc);
        yz[S.roff + j] = acc;
        return;
    }
    if (jl < nj) {
        float* u = gstage + jl;
        stream_direction(S.seed, (uint32_t)S.qctr, (uint32_t)rnd, (uint32_t)j, S.d, ap, pole, u, GEN_STRIDE);
        double acc = 0.0;
        for (int l = 0; l < S.d; ++l) acc = __fma_rn((double)u[l * GEN_STRIDE], z[l], acc);
        yz[S.roff + j] = acc;
    }
    __syncthreads();
    // rows j0 .. j0 + nj - 1 of this query are contiguous in U
    float* base = U + S.uoff + (int64_t)j0 * S.ldx;
    const int ldx = S.ldx, total = nj * ldx;
    for (int e = jl; e < total; e += GEN_NT) {
        const int r = e / ldx, l = e - r * ldx;
        base[e] = l < S.d ? gstage[l * GEN_STRIDE + r] : 0.0f;
    }
}

__global__ void __launch_bounds__(GEN_NT) k_gen(const TaskDev* __restrict__ tasks, const SlotDev* __restrict__ slots,
                                                const float* __restrict__ poles, const float* __restrict__ poles1,
                                                const double* __restrict__ z64, float* __restrict__ U,
                                                double* __restrict__ yz, ResDev* __restrict__ res, int round0, int stage_d)
{
    extern __shared__ float gstage[];
    const TaskDev T = tasks[blockIdx.x];
    const SlotDev& S = slots[T.slot];
    // launch-wide round, or (round0 < 0) the slot's own round with its pole buffer by parity
    const int rnd = round0 >= 0 ? round0 : S.round;
    const float* pcur = round0 >= 0 ? poles : ((rnd & 1) ? poles1 : poles);
    gen_rows(S, T.j0, T.nj, rnd, pcur + S.zoff32, z64, U, yz, res, stage_d, gstage);
}

// The end of round round0 and the start of the next for slots of at most GEN_NT directions, one CTA per slot: the
// round minimum and the pole update (k_argmin's rules), then, unless that was the slot's last round, its next
// directions around the new pole (k_gen's).  One launch where two of them each cost a short call a launch gap per
// round.
__global__ void __launch_bounds__(GEN_NT) k_next(SlotDev* __restrict__ slots, const int32_t* __restrict__ slot_list,
                                                 const float* __restrict__ pcur, float* __restrict__ pnext,
                                                 const double* __restrict__ z64, float* __restrict__ U,
                                                 double* __restrict__ yz, ResDev* __restrict__ res, int round0, int stage_d)
{
    extern __shared__ float gstage[];
    __shared__ double sv[GEN_NT / 32];
    __shared__ int64_t sc[GEN_NT / 32];
    __shared__ int sj[GEN_NT / 32];
    SlotDev& S = slots[slot_list[blockIdx.x]];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, m = S.m;
    const bool hd = (S.kind == 0);
    double bv = INFINITY;
    int64_t bc = INT64_MAX;
    int bj = INT32_MAX;
    if (tid < m) {
        const ResDev r = res[S.roff + tid];
        if (hd ? (r.count < bc) : (r.depth < bv)) {
            bv = r.depth;
            bc = r.count;
            bj = tid;
        }
    }
    auto merge = [&](double ov, int64_t oc, int oj) {
        const bool better = hd ? (oc < bc || (oc == bc && oj < bj)) : (ov < bv || (ov == bv && oj < bj));
        if (better) {
            bv = ov;
            bc = oc;
            bj = oj;
        }
    };
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const double ov = __shfl_xor_sync(0xFFFFFFFFu, bv, o);
        const int64_t oc = __shfl_xor_sync(0xFFFFFFFFu, bc, o);
        const int oj = __shfl_xor_sync(0xFFFFFFFFu, bj, o);
        merge(ov, oc, oj);
    }
    if (lane == 0) {
        sv[w] = bv;
        sc[w] = bc;
        sj[w] = bj;
    }
    const int64_t cmin = S.cmin;
    const double dmin = S.dmin;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < GEN_NT / 32; ++i) merge(sv[i], sc[i], sj[i]);   // every thread gets the same minimum
    const bool take = hd ? (bc < cmin) : (bv < dmin);
    const float* src = take ? U + S.uoff + (int64_t)bj * S.ldx : pcur + S.zoff32;
    for (int l = tid; l < S.ldx; l += GEN_NT) pnext[S.zoff32 + l] = src[l];
    const bool last = round0 == S.r - 1;
    if (tid == 0) {
        const int best = take ? round0 * m + bj : S.best;
        if (take) {
            S.dmin = bv;
            S.cmin = bc;
            S.best = best;
        }
        if (S.choice_out) S.choice_out[round0] = take ? bj : -1;
        if (last) {
            if (S.depth_out) S.depth_out[0] = take ? bv : dmin;
            if (S.count_out) S.count_out[0] = hd ? (take ? bc : cmin) : -1;
            if (S.best_out) S.best_out[0] = best;
        }
    }
    if (last) return;
    __syncthreads();   // the new pole is written, and the old directions are no longer read
    gen_rows(S, 0, m, round0 + 1, pnext + S.zoff32, z64, U, yz, res, stage_d, gstage);
}

// directions of up to max_ldx dims are staged in shared memory (up to GEN_STAGE_MAX bytes)
static int gen_stage_d(int max_ldx)
{
    const size_t per_dim = sizeof(float) * GEN_STRIDE;
    return (size_t)max_ldx * per_dim > GEN_STAGE_MAX ? (int)(GEN_STAGE_MAX / per_dim) : max_ldx;
}

cudaError_t launch_next(SlotDev* slots, const int32_t* slot_list, int nlist, const float* poles_cur, float* poles_next,
                        const double* z64, float* U, double* yz, ResDev* res, int round0, int max_ldx, cudaStream_t st)
{
    if (nlist <= 0) return cudaSuccess;
    const int stage_d = gen_stage_d(max_ldx);
    const size_t smem = (size_t)stage_d * sizeof(float) * GEN_STRIDE;
    static SmemLimit limit;
    const cudaError_t e = limit.raise(k_next);
    if (e != cudaSuccess) return e;
    k_next<<<nlist, GEN_NT, smem, st>>>(slots, slot_list, poles_cur, poles_next, z64, U, yz, res, round0, stage_d);
    return cudaGetLastError();
}

static cudaError_t gen_launch(const TaskDev* tasks, int ntasks, const SlotDev* slots, const float* p0,
                              const float* p1, const double* z64, float* U, double* yz, ResDev* res, int round0,
                              int max_ldx, cudaStream_t st)
{
    if (ntasks <= 0) return cudaSuccess;
    const int stage_d = gen_stage_d(max_ldx);
    const size_t smem = (size_t)stage_d * sizeof(float) * GEN_STRIDE;
    static SmemLimit limit;
    const cudaError_t e = limit.raise(k_gen);
    if (e != cudaSuccess) return e;
    k_gen<<<ntasks, GEN_NT, smem, st>>>(tasks, slots, p0, p1, z64, U, yz, res, round0, stage_d);
    return cudaGetLastError();
}

cudaError_t launch_gen(const TaskDev* tasks, int ntasks, const SlotDev* slots, const float* poles_cur,
                       const double* z64, float* U, double* yz, ResDev* res, int round0, int max_ldx, cudaStream_t st)
{
    return gen_launch(tasks, ntasks, slots, poles_cur, nullptr, z64, U, yz, res, round0, max_ldx, st);
}

cudaError_t launch_gen_slotround(const TaskDev* tasks, int ntasks, const SlotDev* slots, const float* poles0,
                                 const float* poles1, const double* z64, float* U, double* yz, ResDev* res,
                                 int max_ldx, cudaStream_t st)
{
    return gen_launch(tasks, ntasks, slots, poles0, poles1, z64, U, yz, res, -1, max_ldx, st);
}

// y_z = u'z in FP64 for caller-supplied directions (debug path)
__global__ void k_yz_only(const TaskDev* __restrict__ tasks, const SlotDev* __restrict__ slots,
                          const double* __restrict__ z64, const float* __restrict__ U, double* __restrict__ yz)
{
    const TaskDev T = tasks[blockIdx.x];
    const int jl = threadIdx.x;
    if (jl >= T.nj) return;
    const SlotDev& S = slots[T.slot];
    const int j = T.j0 + jl;
    const float* u = U + S.uoff + (int64_t)j * S.ldx;
    double acc = 0.0;
    const double* z = z64 + S.zoff64;
    for (int l = 0; l < S.d; ++l) acc = __fma_rn((double)u[l], z[l], acc);
    yz[S.roff + j] = acc;
}

cudaError_t launch_yz_only(const TaskDev* tasks, int ntasks, const SlotDev* slots, const double* z64, const float* U,
                           double* yz, cudaStream_t st)
{
    if (ntasks <= 0) return cudaSuccess;
    k_yz_only<<<ntasks, 128, 0, st>>>(tasks, slots, z64, U, yz);
    return cudaGetLastError();
}

// caller-supplied directions (n_slots x m x d, dense) into the padded U rows
__global__ void k_scatter_dirs(const SlotDev* __restrict__ slots, int nslots, int m, int d, const float* __restrict__ Uin,
                               float* __restrict__ U)
{
    const int s = blockIdx.x;
    if (s >= nslots) return;
    const SlotDev& S = slots[s];
    for (int e = threadIdx.x; e < m * S.ldx; e += blockDim.x) {
        const int j = e / S.ldx, l = e - j * S.ldx;
        U[S.uoff + e] = (l < d) ? Uin[((int64_t)s * m + j) * d + l] : 0.0f;
    }
}

cudaError_t launch_scatter_dirs(const SlotDev* slots, int nslots, int m, int d, const float* Uin, float* U,
                                cudaStream_t st)
{
    if (nslots <= 0) return cudaSuccess;
    k_scatter_dirs<<<nslots, 128, 0, st>>>(slots, nslots, m, d, Uin, U);
    return cudaGetLastError();
}

__global__ void k_debug_dirs(uint64_t seed, int q, int round0, int m, int d, float alpha, const float* pole,
                             float* U)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    stream_direction(seed, (uint32_t)q, (uint32_t)round0, (uint32_t)j, d, alpha_power(alpha, round0), pole,
                     U + (int64_t)j * d, 1);
}

cudaError_t launch_debug_dirs(uint64_t seed, int q, int round0, int m, int d, float alpha, const float* pole,
                              float* U, cudaStream_t st)
{
    if (m <= 0) return cudaSuccess;
    k_debug_dirs<<<(m + 127) / 128, 128, 0, st>>>(seed, q, round0, m, d, alpha, pole, U);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// halfspace counts, FP32 SIMT projection + exact recheck of the near-tie band
// ---------------------------------------------------------------------------

// One CTA takes up to HD_TJ consecutive (query, direction) rows of one request and walks the points in chunks of
// HD_PC.  Bound by the FMA pipe and the register ports in front of it; the projection is k_keys' register tile
// (16 points x 8 directions per thread as packed FMAs, fma2 / dup2).  Each accumulator starts at -u'z, so the chain
// ends in t = u'x - u'z itself, and the comparison with the band costs three slots per pair: packed t + b and
// b - t, whose sign bits (t < -b, t > b) are shifted into one word per direction and counted.  Pairs with neither
// bit set are near ties and take the exact test.  The directions stay in shared memory; the points come 16 dims at
// a time, the next 16 in flight in registers.
// Measured at d = 50, n = 100,000, 100 queries of 100 directions: 9.28 ms per round with 4 x 4 scalar outputs per
// thread, 5.11 ms with this tile, 2.78 ms with the points also split (hd_parts), 2.57 ms with rows' own bounds (own_z):
// half of the FMA peak.
constexpr int HD_NT = 128;
constexpr int HD_TJ = HD_ROWS;   // rows (query, direction) per CTA
constexpr int HD_PC = 256;       // points per chunk
constexpr int HD_K = 16;         // dims per staging step

// Parts the points are split into.  Two CTAs share an SM, and a launch of few tasks leaves SMs empty or ends in a
// wave that is nearly empty: below eight waves of tasks the points are split into as many parts as give about
// eight waves, each of at least HD_MIN_CHUNKS chunks (a part stages its directions again and meets the others in
// the result cells).  Measured, 157 tasks at d = 50, n = 100,000: 5.11 ms per round unsplit, 2.78 ms in 16 parts.
constexpr int HD_WAVE = 2 * 152, HD_MIN_CHUNKS = 4;
static int hd_parts(int ntasks, int64_t max_n)
{
    if (ntasks >= 8 * HD_WAVE) return 1;
    const int64_t chunks = (max_n + HD_PC - 1) / HD_PC, want = (8 * HD_WAVE + ntasks - 1) / ntasks;
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, chunks / HD_MIN_CHUNKS));
}

// Exact sign of u'(x_i - z) of one near tie; a call of its own, so the register tile's code stays small.
__device__ __noinline__ int hd_exact(const DsDev& D, const float* u, int64_t i, const double* z, int* err)
{
    if (D.X64) return exact_sign<double>(u, 1, D.X64 + i * D.d, z, D.d, err);
    return exact_sign<float>(u, 1, D.X32 + i * D.ldx, z, D.d, err);
}

__global__ void __launch_bounds__(HD_NT, 2) k_hd_simt(const TaskDev* __restrict__ tasks,
                                                      const SlotDev* __restrict__ slots,
                                                      const DsDev* __restrict__ dsets, const float* __restrict__ U,
                                                      const double* __restrict__ yz, const double* __restrict__ z64,
                                                      ResDev* __restrict__ res, int64_t* __restrict__ band_out, int* err)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ int64_t r_uoff[HD_TJ], r_zoff[HD_TJ], r_roff[HD_TJ];
    __shared__ int r_slot[HD_TJ];
    __shared__ unsigned long long c_lt[HD_TJ], c_gt[HD_TJ];
    __shared__ float r_ny[HD_TJ], r_gz[HD_TJ];
    __shared__ unsigned zmax_bits, zmin_bits;
    const TaskDev T = tasks[blockIdx.x];
    const DsDev D = dsets[slots[T.slot].ds];
    const int ldx = D.ldx, d = D.d, dp4 = (d + 3) & ~3;
    const int64_t n = D.n;
    float* Xs = sm;                              // 2 x HD_K x HD_PC: [dim][point]
    float* bS = Xs + 2 * HD_K * HD_PC;           // 2 x HD_PC: band bound of each point of the chunk
    float* Us = bS + 2 * HD_PC;                  // dp4 x HD_TJ: [dim][row]
    // this CTA's points: part blockIdx.y of nparts, in whole chunks
    const int64_t nch = (n + HD_PC - 1) / HD_PC, per = (nch + gridDim.y - 1) / gridDim.y;
    const int nparts = (int)((nch + per - 1) / per);
    const int64_t ibeg = (int64_t)blockIdx.y * per * HD_PC;
    if (ibeg >= n) return;
    const int64_t iend = ibeg + per * HD_PC < n ? ibeg + per * HD_PC : n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (tid == 0) {
        zmax_bits = 0u;
        zmin_bits = 0x7F800000u;
    }
    // norms of 32 points, for the choice of the band below: every warp reads the same ones
    const float xs32 = D.xnorm[lane * (n - 1) / 31];
    const float gamma = band_gamma_fp32(d);
    __syncthreads();
    if (tid < HD_TJ) {
        const int r = tid;
        c_lt[r] = c_gt[r] = 0ull;
        r_ny[r] = r_gz[r] = 0.0f;
        r_slot[r] = -1;
        if (r < T.nj) {
            const int m = slots[T.slot].m;
            const int gg = T.j0 + r, qs = gg / m, j = gg - qs * m;   // rows may run into the request's next queries
            const SlotDev& S = slots[T.slot + qs];
            r_slot[r] = T.slot + qs;
            r_uoff[r] = S.uoff + (int64_t)j * ldx;
            r_zoff[r] = S.zoff64;
            r_roff[r] = S.roff + j;
            r_ny[r] = -(float)yz[S.roff + j];
            r_gz[r] = gamma * S.znorm;
            atomicMax(&zmax_bits, __float_as_uint(S.znorm));   // norms are not negative
            atomicMin(&zmin_bits, __float_as_uint(S.znorm));
        }
    }
    __syncthreads();
    for (int e = tid; e < HD_TJ * (dp4 / 4); e += HD_NT) {
        const int r = e & (HD_TJ - 1), l = (e / HD_TJ) * 4;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < T.nj) v = *reinterpret_cast<const float4*>(U + r_uoff[r] + l);
        Us[l * HD_TJ + r] = v.x;
        Us[(l + 1) * HD_TJ + r] = v.y;
        Us[(l + 2) * HD_TJ + r] = v.z;
        Us[(l + 3) * HD_TJ + r] = v.w;
    }
    // The band of a pair is gamma (|x| + |z|).  With the largest |z| of the rows it is one bound per point, three slots
    // a pair; that suits rows whose norms are alike, or small beside the points'.  A query far from the rest would
    // widen its neighbours' bands to a large share of all points, each of them an exact test, so there every row
    // takes its own |z| (one more packed add).  Measured, n = 100,000, d = 50, 100 queries, 5 rounds of 100 directions:
    // 13.9 ms with normal queries; with five of them 10^5 times as far out 350 ms under one bound, 13.8 ms with their
    // own; heavy-tailed (Student t) queries, 20 rounds, 55.8 -> 51.5 ms.
    const float zmax = __uint_as_float(zmax_bits);
    const bool own_z = zmax > 2.0f * __uint_as_float(zmin_bits) &&
                       __popc(__ballot_sync(0xFFFFFFFFu, 4.0f * xs32 >= zmax)) < 16;   // the same in every warp
    const float gz = own_z ? 0.0f : gamma * zmax;

    // staging: thread tid takes point rows tid and tid + 128 of the chunk (transposed stores free of conflicts)
    float4 xg[2][HD_K / 4];
    float xn[2];
    auto fetch = [&](int64_t i0, int k0) {
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int64_t i = i0 + tid + p * HD_NT;
            const float* xr = D.X32 + i * ldx + k0;
            if (k0 == 0) xn[p] = i < n ? D.xnorm[i] : 0.0f;
#pragma unroll
            for (int h = 0; h < HD_K / 4; ++h) {
                xg[p][h] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i < n && k0 + 4 * h < dp4) xg[p][h] = *reinterpret_cast<const float4*>(xr + 4 * h);
            }
        }
    };
    auto stage = [&](int b, int cb, bool first) {
        float* xs = Xs + b * HD_K * HD_PC + tid;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            if (first) bS[cb * HD_PC + tid + p * HD_NT] = fmaf(gamma, xn[p], gz);
#pragma unroll
            for (int h = 0; h < HD_K / 4; ++h) {
                xs[(4 * h) * HD_PC + p * HD_NT] = xg[p][h].x;
                xs[(4 * h + 1) * HD_PC + p * HD_NT] = xg[p][h].y;
                xs[(4 * h + 2) * HD_PC + p * HD_NT] = xg[p][h].z;
                xs[(4 * h + 3) * HD_PC + p * HD_NT] = xg[p][h].w;
            }
        }
    };
    // this thread's points p0 + 32 a + {0..3}, a = 0..3, and rows q0 + 16 c + {0..3}, c = 0, 1
    const int p0 = (warp & 1) * 128 + (lane & 7) * 4, q0 = (warp >> 1) * 32 + (lane >> 3) * 4;
    auto row_of = [&](int c) { return q0 + 16 * (c >> 2) + (c & 3); };
    unsigned long long acc[8][8];   // [point pair][row]
    auto reset = [&] {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const unsigned long long y = dup2(r_ny[row_of(c)]);
#pragma unroll
            for (int a = 0; a < 8; ++a) acc[a][c] = y;
        }
    };
    int lt[8], gt[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) lt[c] = gt[c] = 0;

    fetch(ibeg, 0);
    stage(0, 0, true);
    __syncthreads();
    reset();
    int64_t i0 = ibeg;
    int k0 = 0, b = 0, cb = 0;
    for (;;) {
        int64_t ni = i0;
        int nk = k0 + HD_K;
        if (nk >= dp4) {
            nk = 0;
            ni = i0 + HD_PC;
        }
        const bool last_k = nk == 0, more = ni < iend;
        if (more) fetch(ni, nk);
        const int kc = dp4 - k0 < HD_K ? dp4 - k0 : HD_K;
        for (int k4 = 0; k4 < kc; k4 += 4) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float* xs = Xs + (b * HD_K + k4 + e) * HD_PC + p0;
                unsigned long long xv[8];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const ulonglong2 x2 = *reinterpret_cast<const ulonglong2*>(xs + 32 * a);
                    xv[2 * a] = x2.x;
                    xv[2 * a + 1] = x2.y;
                }
                const float* us = Us + (k0 + k4 + e) * HD_TJ + q0;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const float4 u4 = *reinterpret_cast<const float4*>(us + 16 * c);
                    const float uv[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const unsigned long long ud = dup2(uv[h]);
#pragma unroll
                        for (int a = 0; a < 8; ++a) acc[a][4 * c + h] = fma2(ud, xv[a], acc[a][4 * c + h]);
                    }
                }
            }
        }
        if (last_k) {
            // bits 31 - k and 15 - k of w[c]: t < -b and t > b of the thread's k-th point, row c
            unsigned w[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) w[c] = 0u;
            const float* bp = bS + cb * HD_PC + p0;
            if (own_z) {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const unsigned long long g2 = dup2(r_gz[row_of(c)]);
                    unsigned wl = 0u, wg = 0u;
#pragma unroll
                    for (int a = 0; a < 8; ++a) {
                        const unsigned long long bz =
                            add2(*reinterpret_cast<const unsigned long long*>(bp + 32 * (a >> 1) + 2 * (a & 1)), g2);
                        const unsigned long long sl = add2(bz, acc[a][c]),
                                                 sg = fma2(acc[a][c], 0xBF800000BF800000ull, bz);
                        wl = __funnelshift_l((unsigned)sl, wl, 1);
                        wl = __funnelshift_l((unsigned)(sl >> 32), wl, 1);
                        wg = __funnelshift_l((unsigned)sg, wg, 1);
                        wg = __funnelshift_l((unsigned)(sg >> 32), wg, 1);
                    }
                    w[c] = wl << 16 | wg;
                }
            } else {
#pragma unroll
                for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const ulonglong2 b2 = *reinterpret_cast<const ulonglong2*>(bp + 32 * a);
                        const unsigned long long bv[2] = {b2.x, b2.y};
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                // pass 0: b + t, negative where t < -b; pass 1: b - t, negative where t > b
                                const unsigned long long s =
                                    pass == 0 ? add2(bv[h], acc[2 * a + h][c])
                                              : fma2(acc[2 * a + h][c], 0xBF800000BF800000ull, bv[h]);
                                w[c] = __funnelshift_l((unsigned)s, w[c], 1);
                                w[c] = __funnelshift_l((unsigned)(s >> 32), w[c], 1);
                            }
                    }
                }
            }
            // points of this thread that exist, first point in bit 15
            unsigned vm = 0xFFFFu;
            if (i0 + HD_PC > n) {
                vm = 0u;
#pragma unroll
                for (int k = 0; k < 16; ++k) vm |= (unsigned)(i0 + p0 + 32 * (k >> 2) + (k & 3) < n) << (15 - k);
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const unsigned l = (w[c] >> 16) & vm, g = w[c] & vm;
                lt[c] += __popc(l);
                gt[c] += __popc(g);
                unsigned cand = vm & ~(l | g);
                const int r = row_of(c);
                if (r >= T.nj) cand = 0u;
                while (cand) {
                    const int k = 31 - __clz(cand);
                    cand &= ~(1u << k);
                    const int pk = 15 - k;
                    const int sgn = hd_exact(D, U + r_uoff[r], i0 + p0 + 32 * (pk >> 2) + (pk & 3),
                                             z64 + r_zoff[r], err);
                    lt[c] += sgn < 0;
                    gt[c] += sgn > 0;
                    if (band_out) atomicAdd((unsigned long long*)&band_out[r_slot[r]], 1ull);
                }
            }
            if (more) reset();
            cb ^= 1;
        }
        if (!more) break;
        stage(b ^ 1, cb, nk == 0);   // the buffer whose readers passed the last barrier
        __syncthreads();
        b ^= 1;
        i0 = ni;
        k0 = nk;
    }
    // the eight point lanes of a direction hold parts of its counts, and so do the two point warps
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        unsigned long long l = (unsigned)lt[c], g = (unsigned)gt[c];
#pragma unroll
        for (int o = 4; o >= 1; o >>= 1) {
            l += __shfl_xor_sync(0xFFFFFFFFu, l, o);
            g += __shfl_xor_sync(0xFFFFFFFFu, g, o);
        }
        if ((lane & 7) == 0) {
            atomicAdd(&c_lt[row_of(c)], l);
            atomicAdd(&c_gt[row_of(c)], g);
        }
    }
    __syncthreads();
    if (tid < T.nj) {
        long long l = (long long)c_lt[tid], g = (long long)c_gt[tid];
        ResDev* cell = res + r_roff[tid];
        if (nparts > 1) {
            // counts of the parts meet in the result cell (zeroed with the directions): #(t > 0) in its count,
            // #(t < 0) below the parts that have arrived in its depth; the last one forms the result
            unsigned long long* cl = reinterpret_cast<unsigned long long*>(&cell->depth);
            unsigned long long* cg = reinterpret_cast<unsigned long long*>(&cell->count);
            atomicAdd(cg, (unsigned long long)g);
            __threadfence();
            const unsigned long long was = atomicAdd(cl, (1ull << HD_PART_SHIFT) + (unsigned long long)l);
            if ((int)(was >> HD_PART_SHIFT) != nparts - 1) return;
            __threadfence();
            l += (long long)(was & ((1ull << HD_PART_SHIFT) - 1));
            g = (long long)atomicAdd(cg, 0ull);
        }
        const int64_t le = n - g, ge = n - l;
        const int64_t c = le < ge ? le : ge;
        *cell = ResDev{(double)c / (double)n, c};
    }
}

cudaError_t launch_hd_simt(const TaskDev* tasks, int ntasks, int max_ldx, int64_t split_n, const SlotDev* slots,
                               const DsDev* ds, const float* U, const double* yz, const double* z64, ResDev* res,
                               int64_t* band_out, int* err, cudaStream_t st)
{
    if (ntasks <= 0) return cudaSuccess;
    const size_t smem = sizeof(float) * ((size_t)HD_TJ * max_ldx + 2 * HD_K * HD_PC + 2 * HD_PC);
    static SmemLimit limit;
    const cudaError_t e = limit.raise(k_hd_simt);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)ntasks, (unsigned)hd_parts(ntasks, split_n));
    k_hd_simt<<<grid, HD_NT, smem, st>>>(tasks, slots, ds, U, yz, z64, res, band_out, err);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// round minimum, strict update of D_min and of the pole (Alg. 1 steps 4-6)
// ---------------------------------------------------------------------------

__global__ void k_argmin(SlotDev* __restrict__ slots, const int32_t* __restrict__ slot_list, int nlist,
                         const float* __restrict__ U, const ResDev* __restrict__ res, float* __restrict__ pa,
                         float* __restrict__ pb, int round_arg)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= nlist) return;
    SlotDev& S = slots[slot_list[w]];
    // launch-wide round (pa = current poles, pb = next), or the slot's own round (pa even, pb odd)
    const int round0 = round_arg >= 0 ? round_arg : S.round;
    const float* poles_cur = round_arg >= 0 ? pa : ((round0 & 1) ? pb : pa);
    float* poles_next = round_arg >= 0 ? pb : ((round0 & 1) ? pa : pb);
    const bool hd = (S.kind == 0);
    // lowest (value, index) over the m directions
    double bv = INFINITY;
    int64_t bc = INT64_MAX;
    int bj = INT32_MAX;
    for (int j = lane; j < S.m; j += 32) {
        const ResDev r = res[S.roff + j];
        const bool better = hd ? (r.count < bc) : (r.depth < bv);
        if (better) {
            bv = r.depth;
            bc = r.count;
            bj = j;
        }
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const double ov = __shfl_xor_sync(0xFFFFFFFFu, bv, o);
        const int64_t oc = __shfl_xor_sync(0xFFFFFFFFu, bc, o);
        const int oj = __shfl_xor_sync(0xFFFFFFFFu, bj, o);
        const bool better = hd ? (oc < bc || (oc == bc && oj < bj)) : (ov < bv || (ov == bv && oj < bj));
        if (better) {
            bv = ov;
            bc = oc;
            bj = oj;
        }
    }
    const bool take = hd ? (bc < S.cmin) : (bv < S.dmin);
    const float* src = take ? U + S.uoff + (int64_t)bj * S.ldx : poles_cur + S.zoff32;
    for (int l = lane; l < S.ldx; l += 32) poles_next[S.zoff32 + l] = src[l];
    if (lane == 0) {
        if (take) {
            S.dmin = bv;
            S.cmin = bc;
            S.best = round0 * S.m + bj;
        }
        if (S.choice_out) S.choice_out[round0] = take ? bj : -1;
        if (round0 == S.r - 1) {
            if (S.depth_out) S.depth_out[0] = S.dmin;
            if (S.count_out) S.count_out[0] = hd ? S.cmin : -1;
            if (S.best_out) S.best_out[0] = S.best;
        }
        if (round_arg < 0) S.round = round0 + 1;
    }
}

cudaError_t launch_argmin(SlotDev* slots, const int32_t* slot_list, int nlist, const float* U, const ResDev* res,
                          const float* poles_cur, float* poles_next, int round0, int last_round, cudaStream_t st)
{
    if (nlist <= 0) return cudaSuccess;
    const int nt = 256;
    const int nb = (nlist * 32 + nt - 1) / nt;
    (void)last_round;
    k_argmin<<<nb, nt, 0, st>>>(slots, slot_list, nlist, U, res, const_cast<float*>(poles_cur), poles_next, round0);
    return cudaGetLastError();
}

cudaError_t launch_argmin_slotround(SlotDev* slots, const int32_t* slot_list, int nlist, const float* U,
                                   const ResDev* res, float* poles0, float* poles1, cudaStream_t st)
{
    if (nlist <= 0) return cudaSuccess;
    const int nt = 256;
    const int nb = (nlist * 32 + nt - 1) / nt;
    k_argmin<<<nb, nt, 0, st>>>(slots, slot_list, nlist, U, res, poles0, poles1, -1);
    return cudaGetLastError();
}

}  // namespace rrs
