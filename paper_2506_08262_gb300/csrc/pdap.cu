// Projection depth D_P and asymmetric projection depth D_AP (Sec. 2) for a block
// of directions: y_i = u'x_i in FP32, exact order statistics (median, MAD,
// MAD_+) of the FP32 keys, whose points a second kernel (k_pdap_finish)
// re-projects in FP64 to form the depth.
//
// The default selection kernels are in pdap_select.cu; this file holds the kernel
// with its keys in shared memory (k_pdap2), the keys kernels, the FP64 finish and
// the launch of a selection.  k_pdap2 runs for a few directions on a long array
// and where rrs_select_kernel or the autotuner ask for 1, 2 or 4 directions per CTA.
//
// One CTA handles G <= 4 directions with the G*n keys resident in shared memory,
// or (allocation-free entry point, d > 16, n beyond what shared memory holds)
// recomputed from X at every pass; the arithmetic is the same throughout, and
// so are the values.  The whole CTA projects (pass A: every point on the G
// directions, keys stored, each added to a 2048-bucket histogram over
// u'c +- 5 sigma_u, bucket = monotone FP32 map of the key).  Then the CTA
// splits into G groups of (CTA threads)/G, one per direction, each synchronising
// on its own named barrier, so the directions never wait for one another:
//   median  find the buckets of the median ranks, gather their keys (and, for
//           D_AP, the keys of the buckets expected to hold the MAD_+ ranks),
//           rank them exactly;
//   D_P     histogram of |y - med|, gather the MAD buckets, rank (MAD).
// Bucket maps are monotone, so every bucket holds a contiguous run of ranks
// and the gathered keys contain the wanted order statistics.  When a run holds
// more keys than the gather buffer, or the D_AP guess of the positive count
// was wrong, the group falls back to an iterated bucket selection over its
// keys.  No per-element work uses FP64.
#include <cuda_runtime.h>
#include <float.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "packed_fma.cuh"
#include "pdap_common.cuh"
#include "rrs_internal.h"

namespace rrs {
namespace {

constexpr int NT = 512;              // threads per CTA for G = 1, 2 (two CTAs per SM)
constexpr int NT4 = 1024;            // threads per CTA for G = 4 (one CTA per SM)
template <int G>
__host__ __device__ constexpr int cta_threads()
{
    return G == 4 ? NT4 : NT;
}
constexpr int MAXG = 4;
// Stride of the resident keys of one direction in shared memory: n rounded up to 32 floats (128 bytes)
__host__ __device__ constexpr int pdap_key_stride(int n) { return (n + 31) & ~31; }

// Per-direction constants and per-group scratch: after the projection pass,
// group g (CTA threads / G) works on direction g alone and synchronises with
// the named barrier 1 + g, so the directions of a CTA never wait for each other.
struct Ctl {
    float lo_b[MAXG], sc_y[MAXG];      // bucket map of the keys: about (y - lo_b) * sc_y
    float off_y[MAXG];                 // -lo_b * sc_y + 2^23 (bucket_m offset)
    float scale[MAXG];                 // sigma_u (or the radius) of each direction
    int red[MAXG][NWARP];
    float fred[MAXG][2 * NWARP];
    int fill[MAXG][2];
    int f_b1[MAXG], f_c1[MAXG], f_b2[MAXG], f_c2[MAXG];   // bucket search results
    int fr_b[MAXG][4], fr_c[MAXG][4], fr_h[MAXG][4];      // gfindn: bucket, keys below, keys in it
    float pv1[MAXG], pv2[MAXG];                           // rank pick results
    int pi1[MAXG], pi2[MAXG];                             // their point indices
    int gn[MAXG];
    int gi[MAXG];                                         // smallest index of a tied run (fallback)
};

// One scan of h[0..NB) by the group locating the buckets of NR ranks rk[] (each below the total): for
// each, the bucket, the keys below it and the keys in it.  With PREFIX, h becomes its inclusive prefix
// counts in the same pass.
template <int GS, int NR, bool PREFIX>
__device__ __forceinline__ void gfindn(const Grp<GS>& q, unsigned* h, const int (&rk)[NR], Ctl& C, int (&bo)[NR], int (&co)[NR],
                       int (&ho)[NR])
{
    constexpr int PER = NB / GS;
    const int lane = q.t & 31, w = q.t >> 5;
    int own = 0;
    unsigned v[PER];
    uint4* h4 = reinterpret_cast<uint4*>(h + q.t * PER);
#pragma unroll
    for (int k = 0; k < PER / 4; ++k) {
        const uint4 a = h4[k];
        v[4 * k] = a.x;
        v[4 * k + 1] = a.y;
        v[4 * k + 2] = a.z;
        v[4 * k + 3] = a.w;
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) own += (int)v[k];
    int incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) C.red[q.g][w] = incl;
    q.sync();
    int base = 0;
#pragma unroll
    for (int i = 0; i < GS / 32; ++i) base += i < w ? C.red[q.g][i] : 0;
    int c = base + incl - own;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int hk = (int)v[k];
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            if (c <= rk[j] && rk[j] < c + hk) {
                C.fr_b[q.g][j] = q.t * PER + k;
                C.fr_c[q.g][j] = c;
                C.fr_h[q.g][j] = hk;
            }
        }
        c += hk;
        if (PREFIX) v[k] = (unsigned)c;
    }
    if (PREFIX) {
#pragma unroll
        for (int k = 0; k < PER / 4; ++k) h4[k] = make_uint4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    }
    q.sync();
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        bo[j] = C.fr_b[q.g][j];
        co[j] = C.fr_c[q.g][j];
        ho[j] = C.fr_h[q.g][j];
    }
    q.sync();
}

// 1 / (1 + num / spread) = spread / (spread + num) for num, spread >= 0 (FP64 inputs, exact differences
// of FP32 order statistics).  GB300 issues FP64 at a fraction of the FP32 rate, so the one division is
// done in FP32 (relative error a few 2^-24) whenever both operands and the quotient are safely normal
// FP32 numbers, and in FP64 otherwise.
__device__ __forceinline__ double depth_from(double num, double spread)
{
    if (spread == 0.0) return num == 0.0 ? 1.0 : 0.0;
    const double den = spread + num;
    if (spread >= 1e-30 && den <= 1e30 && spread >= 1e-20 * den)
        return (double)__fdiv_rn((float)spread, (float)den);
    return spread / den;
}

// Key u'x for d <= 16 (DP4 = d rounded up to 4): two sequential FMA chains over the two
// halves of the DP4 dims, added (two independent chains per key).  Keys and y_z are formed
// the same way whatever the group size, so results never depend on it.
template <int DP4>
__device__ __forceinline__ float key_halves(const float* u, const float* x)
{
    float p0 = 0.f, p1 = 0.f;
#pragma unroll
    for (int l = 0; l < DP4 / 2; ++l) p0 = fmaf(u[l], x[l], p0);
#pragma unroll
    for (int l = DP4 / 2; l < DP4; ++l) p1 = fmaf(u[l], x[l], p1);
    return __fadd_rn(p0, p1);
}

// Pass A of k_pdap2 for d <= 16 (D4 = d rounded up to 4, the directions uu in registers): the keys of G
// directions for the points t0, t0 + 1, then step further on, stored and counted in the
// directions' histograms.  Two points per thread: from the dataset's columns Xt (dim l of point i at
// l * colst + i) their coordinates come as one 8-byte load per dim, side by side over the lanes; without columns
// from the padded rows.
template <int G, int D4>
__device__ __forceinline__ void pass_a_pairs(const DsDev& D, int t0, int step, int n, int kst, const float (&uu)[G][D4],
                                             const float (&sc)[G], const float (&of)[G], float* keys, unsigned* hist)
{
    const size_t colst = (size_t)((n + 31) & ~31);
    for (unsigned i = t0; i < (unsigned)n; i += step) {
        const bool two = i + 1 < (unsigned)n;
        float xa[D4], xb[D4];
        if (D.Xt) {
#pragma unroll
            for (int l = 0; l < D4; ++l) {
                float2 v = make_float2(0.f, 0.f);
                if (l < D.d) v = *reinterpret_cast<const float2*>(D.Xt + l * colst + i);
                xa[l] = v.x;
                xb[l] = v.y;
            }
        } else {
            const float4* ra = reinterpret_cast<const float4*>(D.X32 + (int64_t)i * D.ldx);
            const float4* rb = reinterpret_cast<const float4*>(D.X32 + (int64_t)(two ? i + 1 : i) * D.ldx);
#pragma unroll
            for (int c = 0; c < D4 / 4; ++c) {
                const float4 a = ra[c], b = rb[c];
                xa[4 * c] = a.x;
                xa[4 * c + 1] = a.y;
                xa[4 * c + 2] = a.z;
                xa[4 * c + 3] = a.w;
                xb[4 * c] = b.x;
                xb[4 * c + 1] = b.y;
                xb[4 * c + 2] = b.z;
                xb[4 * c + 3] = b.w;
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const float ka = key_halves<D4>(uu[g], xa), kb = key_halves<D4>(uu[g], xb);
            *reinterpret_cast<float2*>(keys + (size_t)g * kst + i) = make_float2(ka, kb);   // kst is even
            atomicAdd(&hist[g * NB + bucket_m(ka, sc[g], of[g])], 1u);
            if (two) atomicAdd(&hist[g * NB + bucket_m(kb, sc[g], of[g])], 1u);
        }
    }
}

// One direction's keys recomputed from the FP32 rows of X with the projection pass's arithmetic (d > 16: one sequential
// FMA chain), so every pass sees the values a resident key would hold.  u: the direction in shared memory, dp4 floats
// (zero padded).
struct KeysRecomputed {
    const float* X;
    const float* u;
    int ldx, dp4;
    __device__ __forceinline__ float get(int i) const
    {
        const float4* xr = reinterpret_cast<const float4*>(X + (int64_t)i * ldx);
        float acc = 0.f;
        for (int l = 0; l < dp4; l += 4) {
            const float4 x = xr[l >> 2];
            const float4 w = *reinterpret_cast<const float4*>(u + l);
            acc = fmaf(w.x, x.x, acc);
            acc = fmaf(w.y, x.y, acc);
            acc = fmaf(w.z, x.z, acc);
            acc = fmaf(w.w, x.w, acc);
        }
        return acc;
    }
    __device__ __forceinline__ float4 get4(int i) const { return make_float4(get(i), get(i + 1), get(i + 2), get(i + 3)); }
};

// D_P's MAD runs, found from the key histogram H of one direction before its median is known.  With the
// median run [ba, bb] (w buckets), let ss be the smallest s with more than k2 keys in the buckets
// [ba - s, bb + s]; the MAD ranks then deviate from the median by more than (ss - 2) and less than
// (ss + w) bucket widths, so their keys lie in two runs L, R at bucket distance about ss on either side.
// The runs taken here add two buckets on each side of that band, which lets the bound check of
// mad_from_runs pass; they are symmetric about (ba + bb) / 2: L = [L0, L1] below the median run and
// R = [R0, R1] above it.  H holds inclusive prefix counts (gfindn with PREFIX).  The runs stay unset (r untouched) when they would
// overlap the median run or the edge buckets, or hold more than cap keys.
template <int GS, class CT>
__device__ __forceinline__ void mad_runs(const Grp<GS>& q, unsigned* H, CT& C, int ba, int bb, int k2, int cap, int4& r,
                         int& cnt1, int& c_in)
{
    if (q.t == 0) C.f_b1[q.g] = NB;
    q.sync();
    // the window count is non-decreasing in s: rounds of GS consecutive values of s, one per thread, so
    // consecutive threads read consecutive prefix counts (no bank conflicts), until one exceeds k2; it
    // does by s = NB - 1, where the window holds all n keys
    int ss = NB;
    for (int s0 = 0; s0 < NB; s0 += GS) {
        const int s = s0 + q.t;
        const int hi = bb + s < NB - 1 ? bb + s : NB - 1, lo = ba - s;
        const int c = (int)H[hi] - (lo >= 1 ? (int)H[lo - 1] : 0);
        if (c > k2) atomicMin(&C.f_b1[q.g], s);
        q.sync();
        ss = C.f_b1[q.g];
        q.sync();
        if (ss < NB) break;
    }
    const int w = bb - ba + 1;
    const int L0 = ba - ss - w - 2, L1 = ba - ss + w + 3, R0 = bb + ss - w - 3, R1 = bb + ss + w + 2;
    if (ss >= w + 4 && L0 >= 1 && R1 <= NB - 2) {
        const int cl = (int)(H[L1] - H[L0 - 1]) + (int)(H[R1] - H[R0 - 1]);
        if (cl <= cap) {
            cnt1 = cl;
            c_in = (int)(H[R0 - 1] - H[L1]);
            r = make_int4(L0, L1, R0, R1);
        }
    }
}

// FP64 projection u'x_i of point i: one sequential FMA chain over the dims, from the FP64 rows when
// the data came in FP64 (the direction generator forms the query's y_z = u'z the same way, so a query
// equal to a data point projects to the same value).  Every product of an FP32 direction component and
// an FP32 (or FP64) coordinate is rounded at most once per added term.
__device__ __forceinline__ double proj64(const DsDev& D, const float* u, int i)
{
    double acc = 0.0;
    if (D.X64) {
        const double* xr = D.X64 + (int64_t)i * D.d;
        for (int l = 0; l < D.d; ++l) acc = __fma_rn((double)u[l], xr[l], acc);
    } else {
        const float* xr = D.X32 + (int64_t)i * D.ldx;
        for (int l = 0; l < D.d; ++l) acc = __fma_rn((double)u[l], (double)xr[l], acc);
    }
    return acc;
}

// FP64 finish of a selection launch: the depth of every direction from its picks (put_picks).  Four
// threads per direction, one per picked point, each forming the point's FP64 projection (proj64: one
// sequential FMA chain over the dims, the order in which the direction generator forms y_z, so a query
// equal to a data point projects to the same value); the first of the four forms
//   D_P  = 1 / (1 + |y_z - med| / MAD),   D_AP = 1 / (1 + (y_z - med)_+ / MAD_+)      (Sec. 2)
// with med the mean of the two median points (even n: the mean of the middle pair, odd n: the point
// twice), and writes it over the picks.  A kernel of its own: with thousands of directions in flight the
// long FP64 latencies overlap, where inside a selection CTA they would hold up the whole group.
__global__ void __launch_bounds__(256) k_pdap_finish(const TaskDev* __restrict__ tasks, int ntasks, int group,
                                                     const SlotDev* __restrict__ slots,
                                                     const DsDev* __restrict__ dsets, const float* __restrict__ U,
                                                     const double* __restrict__ yz, ResDev* __restrict__ res)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int k = (int)(t & 3);
    const int64_t dir = t >> 2;
    const int64_t ti = dir / group;
    const int g = (int)(dir - ti * group);
    bool live = ti < ntasks;
    TaskDev T{};
    if (live) {
        T = tasks[ti];
        live = g < T.nj;
    }
    double y = 0.0;
    int2 a = make_int2(-1, -1), b = make_int2(-1, -1);
    bool ap = false;
    double yzv = 0.0;
    ResDev* cell = nullptr;
    if (live) {
        const SlotDev& S = slots[T.slot];
        const DsDev& D = dsets[T.ds];
        cell = res + S.roff + T.j0 + g;
        a = reinterpret_cast<const int2*>(cell)[0];
        b = reinterpret_cast<const int2*>(cell)[1];
        ap = S.kind == 2;
        yzv = yz[S.roff + T.j0 + g];
        const int sel = k == 0 ? a.x : (k == 1 ? a.y : (k == 2 ? b.x : b.y));
        if (sel >= 0 && sel < D.n) y = proj64(D, U + S.uoff + (int64_t)(T.j0 + g) * D.ldx, sel);
    }
    // every lane of the warp takes part in the shuffles; the four lanes of a direction are adjacent
    const int lane = threadIdx.x & 31, l0 = lane & ~3;
    const double y0 = __shfl_sync(0xFFFFFFFFu, y, l0), y1 = __shfl_sync(0xFFFFFFFFu, y, l0 + 1);
    const double y2 = __shfl_sync(0xFFFFFFFFu, y, l0 + 2), y3 = __shfl_sync(0xFFFFFFFFu, y, l0 + 3);
    if (!live || k != 0) return;
    const int im1 = a.x, im2 = a.y, ip1 = b.x, ip2 = b.y;
    double depth = __longlong_as_double(0x7FF8000000000000LL);   // a failed selection (error flag set)
    if (im1 >= 0 && im2 >= 0) {
        const double med = (y0 + y1) * 0.5;
        if (ap) {
            double madp = 0.0;
            if (ip1 != NOPOS) madp = ip1 >= 0 && ip2 >= 0 ? fmax(((y2 - med) + (y3 - med)) * 0.5, 0.0) : depth;
            depth = depth_from(yzv - med > 0.0 ? yzv - med : 0.0, madp);
        } else if (ip1 >= 0 && ip2 >= 0) {
            depth = depth_from(fabs(yzv - med), (fabs(y2 - med) + fabs(y3 - med)) * 0.5);
        }
    }
    *cell = ResDev{depth, -1};
}

// Exact median / MAD / MAD_+ of one direction's keys y (after the projection pass), by its group q of
// GS threads.  The selection runs on the FP32 keys and yields the points holding the wanted order
// statistics (ties broken by point index), written to the direction's result cell (put_picks);
// k_pdap_finish forms the depth from FP64 projections of those few points and the FP64 y_z.
//   median  the bucket run of ranks k1, k2 (from the key histogram H) is gathered and ranked;
//   D_P     a |y - med| histogram pass, then the gather and ranking of the MAD run;
//   D_AP    in the median's gather pass, the run of the MAD_+ ranks guessed for no key tying the median.
// Runs that overflow the gather buffer fall back to iterated bucket selection.
// The gather pass of select_dir: every key whose raw bucket value lies in the median run [ml, ml + wm]
// moves, with its point index, to (B0, I0); every key in one of the NR2 second runs [l1, l1 + w1],
// [l2, l2 + w2] to (B1, I1), which holds cap1 pairs (ranges of raw values, compared as unsigned
// differences).  Four keys are tested at once with no branch into a mask of eight bits (key k in the median
// run, in a second run); a thread then takes one pass per set bit, so a warp spends on the rare gathered keys
// only as many passes as its busiest thread.  The keys gathered, and so the picks, are those of a test key by
// key.
template <int GS, int NR2, class K>
__device__ __forceinline__ void gather_runs(const Grp<GS>& q, const K& y, int n, float sc, float of, int ml,
                                            unsigned wm, int l1, unsigned w1, int l2, unsigned w2, int* fill,
                                            float* B0, int* I0, float* B1, int* I1, int cap1)
{
    auto in0 = [&](int rv) { return (unsigned)rv - (unsigned)ml <= wm; };
    auto in1 = [&](int rv) {
        bool h = false;
        if (NR2 >= 1) h = (unsigned)rv - (unsigned)l1 <= w1;
        if (NR2 >= 2) h = h | ((unsigned)rv - (unsigned)l2 <= w2);
        return h;
    };
    // one gathered key: set 0 (the median run) or 1 (the second runs)
    auto put = [&](int set, float v, int i) {
        const int pos = atomicAdd(&fill[set], 1);
        if (pos < (set ? cap1 : CAP)) {
            (set ? B1 : B0)[pos] = v;
            (set ? I1 : I0)[pos] = i;
        }
    };
    const int n4 = n & ~3;
    for (int i = 4 * q.t; i < n4; i += 4 * GS) {
        const float4 y4 = y.get4(i);
        const int r0 = bucket_raw(y4.x, sc, of), r1 = bucket_raw(y4.y, sc, of), r2 = bucket_raw(y4.z, sc, of),
                  r3 = bucket_raw(y4.w, sc, of);
        // bit k: key k in the median run; bit 4 + k: key k in a second run
        unsigned mk = (unsigned)in0(r0) | ((unsigned)in0(r1) << 1) | ((unsigned)in0(r2) << 2) |
                      ((unsigned)in0(r3) << 3) | ((unsigned)in1(r0) << 4) | ((unsigned)in1(r1) << 5) |
                      ((unsigned)in1(r2) << 6) | ((unsigned)in1(r3) << 7);
        while (mk) {   // one pass per gathered key of this thread (most threads: none)
            const int b = __ffs(mk) - 1;
            mk &= mk - 1;
            const int k = b & 3;
            const float v = k == 0 ? y4.x : (k == 1 ? y4.y : (k == 2 ? y4.z : y4.w));
            put(b >> 2, v, i + k);
        }
    }
    for (int i = n4 + q.t; i < n; i += GS) {
        const float v = y.get(i);
        const int rv = bucket_raw(v, sc, of);
        if (in0(rv)) put(0, v, i);
        if (NR2 > 0 && in1(rv)) put(1, v, i);
    }
}

template <int GS, class K>
__device__ __forceinline__ void select_dir(const Grp<GS>& q, const K& y, Ctl& C, unsigned* H, float* B0, int* I0,
                                           int n, bool ap, const DsDev& D, int64_t roff, ResDev* __restrict__ res,
                                           int* err)
{
    const int g = q.g;
    float* B1 = B0 + CAP;   // CAP1 entries: MAD_+ guess run (D_AP) or the runs L, R / the MAD run (D_P)
    int* I1 = I0 + CAP;
    const float sc = C.sc_y[g], of = C.off_y[g];
    const int k1 = (n - 1) / 2, k2 = n / 2;
    const int n4 = n & ~3;
    const float qnan = __int_as_float(0x7FC00000);
    constexpr int OFF = 1 << 30;   // a run start no bucket test can reach

    // one histogram scan: the median ranks, and for D_AP the ranks of the MAD_+ run guessed for no key
    // tying the median (for D_P the scan leaves prefix counts for mad_runs)
    const int npos_guess = (n & 1) ? (n - 1) / 2 : n / 2;
    int ba, ca, bb, cb, hb;
    int b3 = 0, c3 = 0, b4 = 0, c4 = 0, h4 = 0;
    if (ap) {
        const int gb = n - npos_guess;
        const int rk[4] = {k1, k2, npos_guess > 0 ? gb + (npos_guess - 1) / 2 : k1,
                           npos_guess > 0 ? gb + npos_guess / 2 : k2};
        int bo[4], co[4], ho[4];
        gfindn<GS, 4, false>(q, H, rk, C, bo, co, ho);
        ba = bo[0], ca = co[0], bb = bo[1], cb = co[1], hb = ho[1];
        b3 = bo[2], c3 = co[2], b4 = bo[3], c4 = co[3], h4 = ho[3];
    } else {
        const int rk[2] = {k1, k2};
        int bo[2], co[2], ho[2];
        gfindn<GS, 2, true>(q, H, rk, C, bo, co, ho);
        ba = bo[0], ca = co[0], bb = bo[1], cb = co[1], hb = ho[1];
    }
    const int c_lo0 = ca, cnt0 = cb + hb - ca;
    int fb = cnt0 > CAP ? 1 : 0;   // 1: fall back for every statistic, 2: only for the spread
    // second gathered set: the buckets of one or two runs [r.x, r.y], [r.z, r.w] (x > y: no run)
    int4 r2 = make_int4(OFF, -OFF, OFF, -OFF);
    int c_lo1 = 0, cnt1 = 0, c_in = 0;
    if (ap && npos_guess > 0) {
        c_lo1 = c3;
        cnt1 = c4 + h4 - c3;
        if (cnt1 > CAP1) fb = 1;
        r2 = make_int4(b3, b4, OFF, -OFF);   // the run [b3, b4]
    } else if (!ap && !fb) {
        mad_runs(q, H, C, ba, bb, k2, CAP1H, r2, cnt1, c_in);
    }
    const bool second = r2.x <= r2.y;
    // D_P runs of more than CAP1 keys go to the histogram area past the NB2 counters of the MAD pick: H is
    // idle from mad_runs until mad_from_runs, which uses only those counters (the |y - med| pass, which
    // clears all of H, needs the runs no more)
    const bool runs_in_h = !ap && second && cnt1 > CAP1;
    float* R1 = runs_in_h ? reinterpret_cast<float*>(H + NB2) : B1;
    int* J1 = runs_in_h ? reinterpret_cast<int*>(H + NB2 + CAP1H) : I1;
    const int cap1 = runs_in_h ? CAP1H : CAP1;
    float m1 = qnan, m2 = qnan, p1 = 0.f, p2 = 0.f;
    int im1 = -1, im2 = -1, ip1 = -1, ip2 = -1;
    int npos = 0;
    if (!fb) {
        if (q.t < 2) C.fill[g][q.t] = 0;
        q.sync();
        // the runs as ranges of raw bucket values (the edge buckets take every value clamped into them)
        const int ml = raw_lo(ba);
        const unsigned wm = (unsigned)raw_hi(bb) - (unsigned)ml;
        const bool two_runs = second && r2.z <= r2.w;
        const int l1 = second ? raw_lo(r2.x) : 0, l2 = two_runs ? raw_lo(r2.z) : 0;
        const unsigned w1 = second ? (unsigned)raw_hi(r2.y) - (unsigned)l1 : 0u;
        const unsigned w2 = two_runs ? (unsigned)raw_hi(r2.w) - (unsigned)l2 : 0u;
        int* fill = &C.fill[g][0];
        if (two_runs)
            gather_runs<GS, 2>(q, y, n, sc, of, ml, wm, l1, w1, l2, w2, fill, B0, I0, R1, J1, cap1);
        else if (second)
            gather_runs<GS, 1>(q, y, n, sc, of, ml, wm, l1, w1, l2, w2, fill, B0, I0, R1, J1, cap1);
        else
            gather_runs<GS, 0>(q, y, n, sc, of, ml, wm, l1, w1, l2, w2, fill, B0, I0, R1, J1, cap1);
        q.sync();
        gpick(q, B0, I0, cnt0, k1 - c_lo0, k2 - c_lo0, C, m1, m2, im1, im2);
        if (ap) {
            // #(y <= med) = #(y <= m1): keys below the run plus gathered keys <= m1
            int c = 0;
            for (int t = q.t; t < cnt0; t += GS) c += (B0[t] <= m1);
            const int nle = c_lo0 + gsum(q, c, C);
            npos = n - nle;
            if (npos > 0) {
                const int s3 = nle + (npos - 1) / 2 - c_lo1, s4 = nle + npos / 2 - c_lo1;
                if (s3 < 0 || s4 >= cnt1)
                    fb = 2;   // the positive count differed from the guess
                else
                    gpick(q, B1, I1, cnt1, s3, s4, C, p1, p2, ip1, ip2);
            }
        } else {
            const float m = __fmul_rn(__fadd_rn(m1, m2), 0.5f);
            if (!(second && mad_from_runs<GS, CAP>(q, R1, J1, cnt1, k1 - c_in, k2 - c_in, m, H, B0, I0, C, p1,
                                                       p2, ip1, ip2))) {
                // |y - med| histogram over [0, 4 sigma_u] (edge bucket clamps), gather, ranks
                float dmax = D.cov ? 4.0f * C.scale[g] : 0.0f;
                const float hard =
                    __fmul_rn(__fadd_rn(D.rc, fabsf(m - C.lo_b[g] - 0.5f * (float)NB / sc)), 1.0001f);
                if (!(dmax > 0.0f) || dmax > hard) dmax = hard;
                if (!(dmax > 0.0f)) dmax = 1.0f;
                const float scd = __fdiv_rn((float)NB, dmax);
                for (int b = q.t; b < NB / 4; b += GS) reinterpret_cast<uint4*>(H)[b] = make_uint4(0u, 0u, 0u, 0u);
                q.sync();
                for (int i = 4 * q.t; i < n4; i += 4 * GS) {
                    const float4 y4 = y.get4(i);
                    atomicAdd(&H[bucket_m(fabsf(__fsub_rn(y4.x, m)), scd, TWO23)], 1u);
                    atomicAdd(&H[bucket_m(fabsf(__fsub_rn(y4.y, m)), scd, TWO23)], 1u);
                    atomicAdd(&H[bucket_m(fabsf(__fsub_rn(y4.z, m)), scd, TWO23)], 1u);
                    atomicAdd(&H[bucket_m(fabsf(__fsub_rn(y4.w, m)), scd, TWO23)], 1u);
                }
                for (int i = n4 + q.t; i < n; i += GS)
                    atomicAdd(&H[bucket_m(fabsf(__fsub_rn(y.get(i), m)), scd, TWO23)], 1u);
                q.sync();
                int da, dca, db, dcb;
                gfind(q, H, k1, k2, C, da, dca, db, dcb);
                const int cntd = dcb + (int)H[db] - dca;
                if (cntd > CAP1) {
                    fb = 2;
                } else {
                    if (q.t == 0) C.fill[g][1] = 0;
                    q.sync();
                    const int bwd = db - da;
                    auto gd = [&](float v, int i) {
                        const float dv = fabsf(__fsub_rn(v, m));
                        const int b = bucket_m(dv, scd, TWO23);
                        if ((unsigned)(b - da) <= (unsigned)bwd) {
                            const int pos = atomicAdd(&C.fill[g][1], 1);
                            if (pos < CAP1) {
                                B1[pos] = dv;
                                I1[pos] = i;
                            }
                        }
                    };
                    for (int i = 4 * q.t; i < n4; i += 4 * GS) {
                        const float4 y4 = y.get4(i);
                        gd(y4.x, i);
                        gd(y4.y, i + 1);
                        gd(y4.z, i + 2);
                        gd(y4.w, i + 3);
                    }
                    for (int i = n4 + q.t; i < n; i += GS) gd(y.get(i), i);
                    q.sync();
                    gpick(q, B1, I1, cntd, k1 - dca, k2 - dca, C, p1, p2, ip1, ip2);
                }
            }
        }
    }

    // ---- fallback: iterated bucket selection over this direction's keys ----------------
    if (fb) {
        float kl = FLT_MAX, kh = -FLT_MAX;
        for (int i = q.t; i < n; i += GS) {
            const float v = y.get(i);
            kl = fminf(kl, v);
            kh = fmaxf(kh, v);
        }
        gminmax(q, kl, kh, C, kl, kh);
        unsigned* HF = H;
        float* BF = B0;   // FB_CAP values: B0 and B1
        int* IF = I0;     // and their indices: I0 and I1
        if (fb == 1)
            gselect(q, [&](int i) { return y.get(i); }, n, k1, k2, kl, kh, HF, BF, IF, C, m1, m2, im1, im2, err);
        if (ap) {
            int c = 0;
            for (int i = q.t; i < n; i += GS) c += (y.get(i) <= m1);
            const int nle = gsum(q, c, C);
            npos = n - nle;
            ip1 = ip2 = -1;
            if (npos > 0)
                gselect(q, [&](int i) { return y.get(i); }, n, nle + (npos - 1) / 2, nle + npos / 2, kl, kh, HF, BF,
                        IF, C, p1, p2, ip1, ip2, err);
        } else {
            const float m = __fmul_rn(__fadd_rn(m1, m2), 0.5f);
            const float dmax = fmaxf(fabsf(__fsub_rn(kl, m)), fabsf(__fsub_rn(kh, m)));
            gselect(q, [&](int i) { return fabsf(__fsub_rn(y.get(i), m)); }, n, k1, k2, 0.0f, dmax, HF, BF, IF, C,
                    p1, p2, ip1, ip2, err);
        }
    }

    // ---- the picks, for the FP64 finish (k_pdap_finish) ---------------------------------------
    if (q.t == 0) put_picks(res + roff + g, im1, im2, ap && npos == 0 ? NOPOS : ip1, ap && npos == 0 ? NOPOS : ip2);
}

// Every live direction of the CTA: group g of cta_threads<G>() / G threads handles direction g alone,
// on its keys in shared memory or (STREAM) recomputed from X.
template <int G, bool STREAM>
__device__ __forceinline__ void select_dirs(Ctl& C, const float* keys, const float* uS, unsigned* hist, float* buf,
                                            int* ibuf, int n, int kst, bool ap, const DsDev& D, int GA,
                                            int64_t roff, ResDev* __restrict__ res, int* err)
{
    constexpr int GS = cta_threads<G>() / G;   // threads per direction group
    const int tid = threadIdx.x;
    const Grp<GS> q{tid / GS, tid % GS};
    const int g = q.g;
    if (g >= GA) return;   // inert direction (no CTA-wide barrier follows)
    unsigned* H = hist + g * NB;
    float* B0 = buf + (size_t)g * (CAP + CAP1);   // two gather runs, contiguous (FB_CAP for the fallback)
    int* I0 = ibuf + (size_t)g * (CAP + CAP1);    // the point index of every gathered key
    const float* u = uS + (size_t)g * D.ldx;
    if (STREAM) {
        const KeysRecomputed y{D.X32, u, D.ldx, (D.d + 3) & ~3};
        select_dir<GS>(q, y, C, H, B0, I0, n, ap, D, roff, res, err);
    } else {
        const KeysArray y{keys + (size_t)g * kst};
        select_dir<GS>(q, y, C, H, B0, I0, n, ap, D, roff, res, err);
    }
}

// G: directions per CTA (compile time); DP4: d rounded up to 4 when <= 16 (the
// directions are then held in registers), 0 for any d; STREAM: no keys in shared
// memory, every pass recomputes them from X (d > 16 only).
// kin: optional precomputed keys, G x npad per task in launch order (launch_pdap_keys), read instead of
// projecting (not with STREAM)
template <int G, int DP4, bool STREAM>
__global__ void __launch_bounds__(cta_threads<G>(), (G >= 4 ? 1 : 2)) k_pdap2(const TaskDev* __restrict__ tasks, const SlotDev* __restrict__ slots,
                                                 const DsDev* __restrict__ dsets, const float* __restrict__ U,
                                                 ResDev* __restrict__ res, int* err, const float* __restrict__ kin)
{
    extern __shared__ __align__(128) float sm[];
    __shared__ Ctl C;
    const TaskDev T = tasks[blockIdx.x];
    const SlotDev& S = slots[T.slot];
    const DsDev D = dsets[T.ds];   // the task carries its dataset row, so both loads go out together
    const int n = (int)D.n, ldx = D.ldx, d = D.d, dp4 = DP4 ? DP4 : ((d + 3) & ~3);
    const bool ap = (S.kind == 2);
    const int tid = threadIdx.x;
    const int npad = (n + 3) & ~3;   // key stride of the keys formed by launch_pdap_keys (kin)
    // key stride in shared memory: a multiple of 32 floats, so every direction's keys start on a 128-byte
    // line and a warp's 32 consecutive keys take one shared-memory wavefront
    const int kst = pdap_key_stride(n);
    float* keys = sm;                                          // G x kst (none when STREAM)
    float* uS = keys + (STREAM ? (size_t)0 : (size_t)G * kst);   // G x ldx
    unsigned* hist = reinterpret_cast<unsigned*>(uS + (size_t)G * ldx);   // G x NB
    float* buf = reinterpret_cast<float*>(hist + (size_t)G * NB);        // G x (CAP + CAP1)
    int* ibuf = reinterpret_cast<int*>(buf + (size_t)G * (CAP + CAP1));  // G x (CAP + CAP1)

    const int GA = T.nj;   // live directions; groups GA..G-1 are inert
    constexpr int NTK = cta_threads<G>();
    for (int e = tid; e < G * ldx; e += NTK) uS[e] = (e / ldx < GA) ? U[S.uoff + (int64_t)T.j0 * ldx + e] : 0.0f;
    for (int e = tid; e < G * NB / 4; e += NTK) reinterpret_cast<uint4*>(hist)[e] = make_uint4(0u, 0u, 0u, 0u);
    // per-direction bucket range: the centre's projection +- 5 sigma_u (sigma_u^2 = u' Cov u),
    // or +- the radius about the centre when no covariance is kept.  Keys outside the range go
    // to the edge buckets, which keeps the bucket map monotone.  One warp per direction: lanes
    // take rows of Cov (the range is a heuristic, so its summation order is free); y_z keeps the
    // keys' own arithmetic (one lane, sequential FMAs).
    // The range warps read their direction from U itself (the values the CTA stages in uS), so the range
    // is formed while the staging goes on, before the one barrier.
    if ((tid >> 5) < G) {
        const int g = tid >> 5, lane = tid & 31;
        float yc = 0.0f, qf = 0.0f;
        if (g < GA && d <= 32) {
            // lane r holds u_r and forms (Cov u)_r from the other lanes' u_c: every load of the warp is
            // independent of the arithmetic, so they go out together
            const float* u = U + S.uoff + (int64_t)(T.j0 + g) * ldx;
            const float ur = lane < d ? u[lane] : 0.0f;
            if (lane < d) yc = __fmul_rn(ur, D.center[lane]);
            if (D.cov) {
                const float* crow = D.cov + lane * d;
                float w = 0.0f;
#pragma unroll 8
                for (int c = 0; c < d; ++c) {
                    const float uc = __shfl_sync(0xFFFFFFFFu, ur, c);
                    if (lane < d) w = fmaf(crow[c], uc, w);
                }
                qf = __fmul_rn(w, ur);
            }
        } else if (g < GA) {   // inert directions keep a zero direction, as staged
            const float* u = U + S.uoff + (int64_t)(T.j0 + g) * ldx;
            for (int r = lane; r < d; r += 32) yc = fmaf(u[r], D.center[r], yc);
            if (D.cov) {
                // lanes stride over the d x d entries, so the covariance loads are independent of each other
                for (int e = lane; e < d * d; e += 32) {
                    const int r = e / d, c2 = e - r * d;
                    qf = fmaf(D.cov[e], __fmul_rn(u[r], u[c2]), qf);
                }
            }
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            yc += __shfl_xor_sync(0xFFFFFFFFu, yc, o);
            qf += __shfl_xor_sync(0xFFFFFFFFu, qf, o);
        }
        if (lane == 0) {
            float half = D.rc * 1.0001f;
            if (D.cov) {
                const float sg = sqrtf(fmaxf(qf, 0.0f));
                if (sg > 0.0f && 5.0f * sg < half) half = 5.0f * sg;
                C.scale[g] = sg;   // kept for the deviation range
            } else {
                C.scale[g] = half;
            }
            if (!(half > 0.0f)) half = fmaxf(fabsf(yc), 1.0f);
            C.lo_b[g] = yc - half;
            C.sc_y[g] = __fdiv_rn((float)NB, __fadd_rn(half, half));
            C.off_y[g] = __fadd_rn(__fmul_rn(-C.lo_b[g], C.sc_y[g]), TWO23);
        }
    }
    __syncthreads();

    // ---- pass A (whole CTA): keys + bucket counts ---------------------------------------
    {
        float of[G], sc[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            of[g] = C.off_y[g];
            sc[g] = C.sc_y[g];
        }
        auto emit = [&](int i, const float (&acc)[G]) {
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if (!STREAM) keys[(size_t)g * kst + i] = acc[g];
                atomicAdd(&hist[g * NB + bucket_m(acc[g], sc[g], of[g])], 1u);
            }
        };
        if (!STREAM && kin) {
            // keys formed by k_keys (same arithmetic as the projection below): count and copy
            const float4* src = reinterpret_cast<const float4*>(kin + (size_t)blockIdx.x * G * npad);
            for (int e = tid; e < G * npad / 4; e += NTK) {
                const int g = e / (npad / 4), i = 4 * (e - g * (npad / 4));
                if (g >= GA) continue;
                const float4 k4 = src[e];
                const float kv[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    if (i + h < n) {
                        keys[(size_t)g * kst + i + h] = kv[h];
                        atomicAdd(&hist[g * NB + bucket_m(kv[h], sc[g], of[g])], 1u);
                    }
                }
            }
        } else if (G == 4 && DP4 > 0) {
            // two adjacent lanes per point, each forming the keys of two directions: the row load is
            // coalesced within the warp and each lane holds only two direction vectors
            constexpr int D4 = DP4 > 0 ? DP4 : 4;
            const int pair = tid & 1;
            float ua[D4], ub[D4];
#pragma unroll
            for (int l = 0; l < D4; ++l) {
                ua[l] = uS[(2 * pair) * ldx + l];
                ub[l] = uS[(2 * pair + 1) * ldx + l];
            }
            float u2[2][D4];
#pragma unroll
            for (int l = 0; l < D4; ++l) {
                u2[0][l] = ua[l];
                u2[1][l] = ub[l];
            }
            const float s2[2] = {sc[2 * pair], sc[2 * pair + 1]}, o2[2] = {of[2 * pair], of[2 * pair + 1]};
            pass_a_pairs<2, D4>(D, 2 * (tid >> 1), NTK, n, kst, u2, s2, o2, keys + (size_t)(2 * pair) * kst,
                                        hist + 2 * pair * NB);
        } else if (DP4 > 0) {
            constexpr int D4 = DP4 > 0 ? DP4 : 4;
            float uu[G][D4];
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int c = 0; c < D4 / 4; ++c) {
                    const float4 u4 = *reinterpret_cast<const float4*>(uS + g * ldx + 4 * c);
                    uu[g][4 * c] = u4.x;
                    uu[g][4 * c + 1] = u4.y;
                    uu[g][4 * c + 2] = u4.z;
                    uu[g][4 * c + 3] = u4.w;
                }
            pass_a_pairs<G, D4>(D, 2 * tid, 2 * NTK, n, kst, uu, sc, of, keys, hist);
        } else {
            for (int i = tid; i < n; i += NTK) {
                const float4* xr = reinterpret_cast<const float4*>(D.X32 + (int64_t)i * ldx);
                float acc[G];
#pragma unroll
                for (int g = 0; g < G; ++g) acc[g] = 0.f;
                for (int l = 0; l < dp4; l += 4) {
                    const float4 x = xr[l >> 2];
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        const float4 u = *reinterpret_cast<const float4*>(uS + g * ldx + l);
                        acc[g] = fmaf(u.x, x.x, acc[g]);
                        acc[g] = fmaf(u.y, x.y, acc[g]);
                        acc[g] = fmaf(u.z, x.z, acc[g]);
                        acc[g] = fmaf(u.w, x.w, acc[g]);
                    }
                }
                emit(i, acc);
            }
        }
    }
    __syncthreads();

    select_dirs<G, STREAM>(C, keys, uS, hist, buf, ibuf, n, kst, ap, D, GA, S.roff + T.j0, res, err);
}

}  // namespace

size_t pdap_smem_bytes(int n, int group, int ldx, bool stream)
{
    const size_t kst = stream ? 0 : (size_t)pdap_key_stride(n);
    return sizeof(float) * ((size_t)group * kst + (size_t)group * ldx) + sizeof(unsigned) * (size_t)group * NB +
           (sizeof(float) + sizeof(int)) * (size_t)group * (CAP + CAP1);
}

size_t pdap_smem_limit()
{
    // opt-in maximum per CTA (227 KB) minus the kernels' static blocks
    return 232448 - sizeof(Ctl) - 64 - 256;
}

// Directions per CTA of the allocation-free call for d > 16: the most of 1, 2, 4 whose keys fit, 0 if none do.  The
// projection pass re-reads X (4 d bytes per point) for every G directions (measured at n = 10,000: d = 50 1.27x,
// d = 150 1.68x faster with G = 4 than G = 2).
int pdap_max_group(int n, int ldx, int m)
{
    int most = 0;
    for (int g = 1; g <= MAXG && g <= m; g *= 2)
        if (pdap_smem_bytes(n, g, ldx) <= pdap_smem_limit()) most = g;
    return most;
}

// Keys of a block of tasks (G directions each, all of one dataset) for every point, as a tiled FP32
// GEMM: keys[(t * G + g) * npad + i] = u_{t,g}'x_i, each key one sequential FMA chain over the dims
// (the selection kernel's own arithmetic for d > 16, and y_z's), so results do not depend on which
// kernel formed the keys.
//
// Bound by the FMA pipe and the register ports in front of it.  CTA tile 128 points x 128 directions, 128
// threads, two CTAs per SM; a thread takes 16 points x 8 directions as 8 point pairs x 8 directions, each
// pair one packed FMA (fma.rn.f32x2: two IEEE FMAs, so every key keeps its chain, in one issue slot).  Per
// dim a thread issues 64 packed FMAs on 6 shared loads; lanes read 16-byte words that are consecutive over
// the 8 point lanes and the 4 direction lanes of a warp, so no load has a bank conflict.  The dims come 16 at
// a time, the next 16 in flight in registers during the FMAs, two staging buffers, one barrier per step; the
// last step runs only the dims that are there (rows are zero-padded to a multiple of 4).
// Measured, 10,000 points x 6,700 directions: d = 50 243 -> 164 us, d = 100 295 us (56% of the FMA peak).
// 8 x 8 outputs per thread, directions duplicated in shared memory: 204 us (shared-memory loads 68% busy);
// duplicated in registers: 181 us; scalar FMAs: 181 us; row-major staging by cp.async: 168 us at best.
constexpr int KT_P = 128, KT_D = 128, KT_K = 16, KT_NT = 128;

__global__ void __launch_bounds__(KT_NT, 2) k_keys(const TaskDev* __restrict__ tasks, int ntasks, int G,
                                                   const SlotDev* __restrict__ slots, const DsDev* __restrict__ dsets,
                                                   const float* __restrict__ U, float* __restrict__ keys, int npad)
{
    __shared__ __align__(16) float Xs[2][KT_K][KT_P];   // [dim][point]
    __shared__ __align__(16) float Us[2][KT_K][KT_D];   // [dim][direction]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const DsDev D = dsets[slots[tasks[0].slot].ds];
    const int n = (int)D.n, ldx = D.ldx, dp4 = (D.d + 3) & ~3;
    const int i0 = blockIdx.x * KT_P, r0 = blockIdx.y * KT_D;
    // staging: thread tid loads the 16 dims of point row tid and of direction row tid (a warp's 32 rows are
    // consecutive, so its transposed stores are free of conflicts)
    const float* urow = nullptr;
    {
        const int r = r0 + tid, t = r / G, g = r - t * G;
        if (t < ntasks && g < tasks[t].nj) {
            const TaskDev T = tasks[t];
            urow = U + slots[T.slot].uoff + (int64_t)(T.j0 + g) * ldx;
        }
    }
    const float* xrow = (i0 + tid < n) ? D.X32 + (int64_t)(i0 + tid) * ldx : nullptr;
    float4 xg[KT_K / 4], ug[KT_K / 4];   // the next step's dims
    auto fetch = [&](int k0) {
#pragma unroll
        for (int h = 0; h < KT_K / 4; ++h) {
            const int l = k0 + 4 * h;
            xg[h] = ug[h] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (xrow && l < dp4) xg[h] = *reinterpret_cast<const float4*>(xrow + l);
            if (urow && l < dp4) ug[h] = *reinterpret_cast<const float4*>(urow + l);
        }
    };
    auto stage = [&](int b) {
#pragma unroll
        for (int h = 0; h < KT_K / 4; ++h) {
            const float xv[4] = {xg[h].x, xg[h].y, xg[h].z, xg[h].w}, uv[4] = {ug[h].x, ug[h].y, ug[h].z, ug[h].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                Xs[b][4 * h + e][tid] = xv[e];
                Us[b][4 * h + e][tid] = uv[e];
            }
        }
    };
    // this thread's points p0 + 32 a + {0..3}, a = 0..3, and directions q0 + 16 c + {0..3}, c = 0, 1
    const int p0 = (lane & 7) * 4, q0 = warp * 32 + (lane >> 3) * 4;
    unsigned long long acc[8][8];   // [point pair][direction]
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[a][c] = 0ull;
    fetch(0);
    stage(0);
    __syncthreads();
    int b = 0;
    for (int k0 = 0; k0 < dp4; k0 += KT_K, b ^= 1) {
        const bool more = k0 + KT_K < dp4;
        if (more) fetch(k0 + KT_K);
        const int kc = dp4 - k0 < KT_K ? dp4 - k0 : KT_K;
        for (int k4 = 0; k4 < kc; k4 += 4) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float* xs = &Xs[b][k4 + e][p0];
                unsigned long long xv[8];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const ulonglong2 x2 = *reinterpret_cast<const ulonglong2*>(xs + 32 * a);
                    xv[2 * a] = x2.x;
                    xv[2 * a + 1] = x2.y;
                }
                const float* us = &Us[b][k4 + e][q0];
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
        if (more) stage(b ^ 1);   // the buffer whose readers passed the last barrier
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int r = r0 + q0 + 16 * (c >> 2) + (c & 3), t = r / G, g = r - t * G;
        if (t >= ntasks || g >= tasks[t].nj) continue;
        float* out = keys + (size_t)r * npad + i0 + p0;
#pragma unroll
        for (int a = 0; a < 4; ++a)
            if (i0 + p0 + 32 * a + 4 <= npad)
                *reinterpret_cast<ulonglong2*>(out + 32 * a) = make_ulonglong2(acc[2 * a][c], acc[2 * a + 1][c]);
    }
}

// Keys for d <= 16 (DP4 = d rounded up to 4) with the selection kernel's own two-half-chain arithmetic
// (key_halves), same layout as k_keys: keys[(t * G + g) * npad + i].  CTA: 256 points x 16 directions,
// one point row in registers per thread, the directions in shared memory, coalesced key writes.
constexpr int KH_P = 256, KH_D = 16;

template <int DP4>
__global__ void __launch_bounds__(KH_P) k_keys_halves(const TaskDev* __restrict__ tasks, int ntasks, int G,
                                                      const SlotDev* __restrict__ slots,
                                                      const DsDev* __restrict__ dsets, const float* __restrict__ U,
                                                      float* __restrict__ keys, int npad)
{
    __shared__ __align__(16) float Us[KH_D][DP4];
    __shared__ int live[KH_D];
    const DsDev D = dsets[slots[tasks[0].slot].ds];
    const int n = (int)D.n, ldx = D.ldx;
    const int r0 = blockIdx.y * KH_D;
    for (int e = threadIdx.x; e < KH_D * DP4; e += KH_P) {
        const int rr = e / DP4, l = e - rr * DP4, r = r0 + rr, t = r / G, g = r - t * G;
        float v = 0.0f;
        if (t < ntasks && g < tasks[t].nj) v = U[slots[tasks[t].slot].uoff + (int64_t)(tasks[t].j0 + g) * ldx + l];
        Us[rr][l] = v;
    }
    if (threadIdx.x < KH_D) {
        const int r = r0 + threadIdx.x, t = r / G, g = r - t * G;
        live[threadIdx.x] = t < ntasks && g < tasks[t].nj;
    }
    __syncthreads();
    const int i = blockIdx.x * KH_P + threadIdx.x;
    if (i >= n) return;
    const float4* xr = reinterpret_cast<const float4*>(D.X32 + (int64_t)i * ldx);
    float xv[DP4];
#pragma unroll
    for (int c = 0; c < DP4 / 4; ++c) {
        const float4 t4 = xr[c];
        xv[4 * c] = t4.x;
        xv[4 * c + 1] = t4.y;
        xv[4 * c + 2] = t4.z;
        xv[4 * c + 3] = t4.w;
    }
#pragma unroll 4
    for (int rr = 0; rr < KH_D; ++rr)
        if (live[rr]) keys[(size_t)(r0 + rr) * npad + i] = key_halves<DP4>(Us[rr], xv);
}

template <int G, int DP4, bool STREAM>
static cudaError_t launch_t(const TaskDev* tasks, int ntasks, size_t smem, const SlotDev* slots, const DsDev* ds,
                            const float* U, const double* yz, ResDev* res, int* err, const float* kin, cudaStream_t st)
{
    static SmemLimit limit;
    const cudaError_t e = limit.raise(k_pdap2<G, DP4, STREAM>);
    if (e != cudaSuccess) return e;
    k_pdap2<G, DP4, STREAM><<<ntasks, cta_threads<G>(), smem, st>>>(tasks, slots, ds, U, res, err, kin);
    return cudaGetLastError();
}

template <int G>
static cudaError_t launch_g(int dp4, const TaskDev* tasks, int ntasks, size_t smem, const SlotDev* slots,
                            const DsDev* ds, const float* U, const double* yz, ResDev* res, int* err, const float* kin,
                            cudaStream_t st)
{
    switch (dp4) {
    case 4: return launch_t<G, 4, false>(tasks, ntasks, smem, slots, ds, U, yz, res, err, kin, st);
    case 8: return launch_t<G, 8, false>(tasks, ntasks, smem, slots, ds, U, yz, res, err, kin, st);
    case 12: return launch_t<G, 12, false>(tasks, ntasks, smem, slots, ds, U, yz, res, err, kin, st);
    case 16: return launch_t<G, 16, false>(tasks, ntasks, smem, slots, ds, U, yz, res, err, kin, st);
    default: return launch_t<G, 0, false>(tasks, ntasks, smem, slots, ds, U, yz, res, err, kin, st);
    }
}

int pdap_dp4_class(int d)
{
    const int dp4 = (d + 3) & ~3;
    return dp4 <= 16 ? dp4 : 0;
}

static cudaError_t launch_select(const TaskDev* tasks, int ntasks, size_t smem, int group, int variant,
                                 const SlotDev* slots, const DsDev* ds, const float* U, const double* yz, ResDev* res,
                                 int* err, cudaStream_t st, const float* kin);

cudaError_t launch_pdap(const TaskDev* tasks, int ntasks, size_t smem, int group, int variant, const SlotDev* slots,
                        const DsDev* ds, const float* U, const double* yz, ResDev* res, int* err, cudaStream_t st,
                        const float* kin)
{
    if (ntasks <= 0) return cudaSuccess;
    const cudaError_t e = launch_select(tasks, ntasks, smem, group, variant, slots, ds, U, yz, res, err, st, kin);
    if (e != cudaSuccess) return e;
    const int64_t threads = (int64_t)ntasks * group * 4;
    const int nt = 256;
    k_pdap_finish<<<(unsigned)((threads + nt - 1) / nt), nt, 0, st>>>(tasks, ntasks, group, slots, ds, U, yz, res);
    return cudaGetLastError();
}

static cudaError_t launch_select(const TaskDev* tasks, int ntasks, size_t smem, int group, int variant,
                                 const SlotDev* slots, const DsDev* ds, const float* U, const double* yz, ResDev* res,
                                 int* err, cudaStream_t st, const float* kin)
{
    if (smem > pdap_smem_limit()) return cudaErrorInvalidValue;
    if (variant & (PDAP_WARP | PDAP_KEYS)) return launch_sel(tasks, ntasks, group, variant, slots, ds, U, res, err, st, kin);
    const int dp4 = variant & ~PDAP_STREAM;
    if (variant & PDAP_STREAM) {
        if (group != PDAP_STREAM_GROUP || dp4 != 0) return cudaErrorInvalidValue;   // d <= 16 has k_select_x
        return launch_t<PDAP_STREAM_GROUP, 0, true>(tasks, ntasks, smem, slots, ds, U, yz, res, err, nullptr, st);
    }
    switch (group) {
    case 1: return launch_g<1>(dp4, tasks, ntasks, smem, slots, ds, U, yz, res, err, kin, st);
    case 2: return launch_g<2>(dp4, tasks, ntasks, smem, slots, ds, U, yz, res, err, kin, st);
    case 4: return launch_g<4>(dp4, tasks, ntasks, smem, slots, ds, U, yz, res, err, kin, st);
    default: return cudaErrorInvalidValue;
    }
}

size_t pdap_keys_bytes(int n, int group, int ntasks)
{
    return sizeof(float) * (size_t)ntasks * group * (((size_t)n + 3) & ~(size_t)3);
}

int pdap_keys_chunk(int n, int d, int group, int64_t ntasks, size_t bytes)
{
    // rows of one keys launch: its grid's y extent, each block a tile of KH_D or KT_D rows
    const int64_t rows = (int64_t)65535 * (pdap_dp4_class(d) ? KH_D : KT_D);
    const int64_t most = std::min<int64_t>(rows / group, (int64_t)(bytes / pdap_keys_bytes(n, group, 1)));
    return (int)std::max<int64_t>(1, std::min(ntasks, most));
}

cudaError_t launch_pdap_keys(const TaskDev* tasks, int ntasks, int group, const SlotDev* slots, const DsDev* ds,
                             const DsDev& ds_host, const float* U, float* keys, cudaStream_t st)
{
    if (ntasks <= 0) return cudaSuccess;
    if (ds_host.n < 1 || ds_host.n > PDAP_MAX_N) return cudaErrorInvalidValue;
    const int npad = (int)((ds_host.n + 3) & ~3LL);
    const int dp4 = pdap_dp4_class(ds_host.d);
    if (dp4 > 0) {
        const dim3 grid((unsigned)((ds_host.n + KH_P - 1) / KH_P), (unsigned)((ntasks * group + KH_D - 1) / KH_D));
        switch (dp4) {
        case 4: k_keys_halves<4><<<grid, KH_P, 0, st>>>(tasks, ntasks, group, slots, ds, U, keys, npad); break;
        case 8: k_keys_halves<8><<<grid, KH_P, 0, st>>>(tasks, ntasks, group, slots, ds, U, keys, npad); break;
        case 12: k_keys_halves<12><<<grid, KH_P, 0, st>>>(tasks, ntasks, group, slots, ds, U, keys, npad); break;
        default: k_keys_halves<16><<<grid, KH_P, 0, st>>>(tasks, ntasks, group, slots, ds, U, keys, npad); break;
        }
        return cudaGetLastError();
    }
    const dim3 grid((unsigned)((ds_host.n + KT_P - 1) / KT_P), (unsigned)((ntasks * group + KT_D - 1) / KT_D));
    k_keys<<<grid, KT_NT, 0, st>>>(tasks, ntasks, group, slots, ds, U, keys, npad);
    return cudaGetLastError();
}

}  // namespace rrs
