// Projection depth D_P and asymmetric projection depth D_AP: the default selection kernels.  k_select_x (d <= 16)
// re-forms the keys from X at both of its passes, k_select reads keys formed once in device memory; both write the
// points holding the order statistics, which k_pdap_finish (pdap.cu) turns into depths.
#include <algorithm>

#define PDAP_BLOCK_GROUPS   // a group of more than one warp is a whole block here (k_select)
#include "packed_fma.cuh"
#include "pdap_common.cuh"
#include "rrs_internal.h"

namespace rrs {
namespace {

// ---------------------------------------------------------------------------------------------
// Selection of one direction by one thread group: k_select (keys in device memory, a block per direction) and
// k_select_x (keys re-formed from X at every pass, a warp per direction)
// ---------------------------------------------------------------------------------------------
// Both take the same four steps per direction and share the code of all but the key source:
//   range    128 keys at evenly spaced points, sorted 32 at a time by one warp: the buckets span their median +- 2 interquartile
//            ranges.  A range from the keys themselves fits every law; one from the covariance is far too wide for
//            heavy tails and costs d^2 products per direction.  It is a heuristic only: keys beyond it are counted
//            in the edge buckets and the bucket map stays monotone, so the picks never depend on it.
//   count    every key into nb buckets (a shared-memory reduction each).
//   runs     the histogram becomes prefix counts; warp searches on them give the bucket run [ba, bb] of the median
//            ranks and the second runs: for D_AP the run of the MAD_+ ranks (guessed for no key tying the median),
//            for D_P the buckets on either side that the MAD ranks must lie in whatever key is the median.
//   gather   every key is tested again and the few (about 1%) in a run are listed with their point indices, in
//            the histogram's memory, which is idle by then.  The picks rank that list.
// A list that would not fit, a run at the edge of the range, or bounds that do not hold once the median is known
// send the direction to the iterated selection (sel_rank).
//
// nb is a power of two chosen by n (sel_buckets): about 16 n / nb keys are listed for D_P (normal data), which must
// fit (nb - 256) / 2 pairs, and each costs its warp some ten instructions; a histogram of nb costs two scans.
__host__ __device__ constexpr int sel_cap0(int nb) { return nb / 16 > 128 ? nb / 16 : 128; }   // median run and pick scratch (pairs)
// shared words per direction: histogram (then the list), median run / pick scratch
__host__ __device__ constexpr int sel_words(int nb) { return nb + 2 * sel_cap0(nb); }
constexpr int SX_G = 8;      // directions of a full k_select_x CTA, each the work of one of its warps between the passes
constexpr int SX_NT = 256;   // its threads: two CTAs per SM, so one's passes run beside the other's warp steps
constexpr size_t SX_SMEM = 110 * 1024;   // its dynamic shared memory, two CTAs per SM

// One direction's bucket map and gather windows, as the passes read them (16-byte parts).
struct __align__(16) SelPar {
    unsigned long long sc2, of2;   // (sc, sc), (of, of): raw bucket value y * sc + of, of = -lo * sc + 2^23
    unsigned long long nrc2;       // (-rc, -rc), rc the raw value the windows are symmetric about
    float w0, w1;                  // listed: |r - rc| <= w0, and second runs ||r - rc| - dd| <= w1 (D_P) or
    float dd;                      // |(r - rc) - dd| <= w1 (D_AP); negative widths: none
    float sc, of, pad;
};

template <int NG>
struct CtlS {
    int red[NG][NWARP / NG];
    float fred[NG][2 * NWARP];
    int fill[NG][2];
    int f_b1[NG], f_c1[NG], f_b2[NG], f_c2[NG];
    float pv1[NG], pv2[NG];
    int pi1[NG], pi2[NG];
    int gn[NG], gi[NG];
    SelPar par[NG];
};

__device__ __forceinline__ float lo_f(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi_f(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }

// Ascending bitonic sort of one value per lane.
__device__ __forceinline__ float warp_sort(float v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const float o = __shfl_xor_sync(0xFFFFFFFFu, v, j);
            const bool up = ((lane & k) == 0) == ((lane & j) == 0);
            v = up ? fminf(v, o) : fmaxf(v, o);
        }
    return v;
}

// Bucket map from RS sampled keys per lane (RS groups of 32): median and interquartile range, the mean of the groups';
// rad bounds |y - centre| (used when the sample has no spread).  A range too narrow for the MAD runs sends the
// direction to the iterated selection, which one such direction per launch makes the launch's tail: with one group
// of 32 and 2 interquartile ranges that was 1 of 2,500 normal directions, with four groups it is below 1 in 10^6.
constexpr int RS = 4;
__device__ __forceinline__ int sel_sample(int n, int lane, int k) { return (int)((int64_t)(RS * lane + k) * (n - 1) / (32 * RS - 1)); }
__device__ __forceinline__ void sel_range(const float (&sample)[RS], float rad, int nb, SelPar& par)
{
    float md = 0.0f, iqr = 0.0f;
#pragma unroll
    for (int k = 0; k < RS; ++k) {
        const float v = warp_sort(sample[k]);
        md += __shfl_sync(0xFFFFFFFFu, v, 16) * (1.0f / RS);
        iqr += (__shfl_sync(0xFFFFFFFFu, v, 23) - __shfl_sync(0xFFFFFFFFu, v, 8)) * (1.0f / RS);
    }
    float half = 2.0f * iqr;
    if (!(half > 0.0f)) half = rad * 2.0002f;
    if (!(half > 0.0f)) half = fmaxf(fabsf(md), 1.0f);
    par.sc = __fdiv_rn((float)nb, half + half);
    par.of = __fadd_rn(__fmul_rn(-(md - half), par.sc), TWO23);
    par.sc2 = dup2(par.sc);
    par.of2 = dup2(par.of);
}

// Inclusive prefix counts of H[0, nb) in place by the group.  Thread t owns nb / GS consecutive buckets, read as
// 16-byte chunks in an order rotated by t, so that 8 consecutive threads touch 8 bank groups; the chunks before
// the rotation's start are summed apart, which gives the running count where the second, ordered sweep begins.
template <int GS, class CT>
__device__ __forceinline__ void sel_prefix(const Grp<GS>& q, unsigned* H, int nb, CT& C)
{
    const int nch = nb / (4 * GS), msk = nch - 1;   // chunks per thread, a power of two
    uint4* h4 = reinterpret_cast<uint4*>(H) + q.t * nch;
    unsigned tail = 0, head = 0;
    const int c0 = q.t & msk;
#pragma unroll 4
    for (int k = 0; k < nch; ++k) {
        const int c = (k + c0) & msk;
        const uint4 a = h4[c];
        const unsigned s = a.x + a.y + a.z + a.w;
        if (c >= c0) tail += s;
        else head += s;
    }
    const int lane = q.t & 31;
    const unsigned own = head + tail;
    unsigned incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    unsigned base = incl - own;
    if (GS > 32) {
        if (lane == 31) C.red[q.g][q.t >> 5] = (int)incl;
        q.sync();
#pragma unroll
        for (int i = 0; i < GS / 32; ++i) base += i < (q.t >> 5) ? (unsigned)C.red[q.g][i] : 0u;
    }
    unsigned run = base + head;
#pragma unroll 4
    for (int k = 0; k < nch; ++k) {
        const int c = (k + c0) & msk;
        if (c == 0) run = base;
        uint4 a = h4[c];
        a.x += run;
        a.y += a.x;
        a.z += a.y;
        a.w += a.z;
        run = a.w;
        h4[c] = a;
    }
    q.sync();
}

// Smallest bucket b with H[b] > rk (H: inclusive prefix counts, rk below the total), by every warp for itself.
__device__ __forceinline__ int sel_find(const unsigned* H, int nb, unsigned rk)
{
    const int lane = threadIdx.x & 31, Q = nb >> 5;
    const int blk = __popc(__ballot_sync(0xFFFFFFFFu, H[(lane + 1) * Q - 1] <= rk));
    int b = blk * Q;
    for (int j = 0; j < Q; j += 32)
        b += __popc(__ballot_sync(0xFFFFFFFFu, j + lane < Q && H[blk * Q + j + lane] <= rk));
    return b;
}

// What the runs step finds (the same in every thread of the group).
struct SelRuns {
    int fb;           // 1: iterated selection for every statistic, 2: for the spread only
    int c_lo0;        // keys below the median run
    int cnt0;         // keys in it
    int cnt;          // keys listed
    int c2;           // rank of a key among all minus its rank in the list: D_AP second run, D_P deviations
    float wm;         // the median run: |r - rc| <= wm
    // D_P: y values that bound the keys left out: between the runs (il, ih), outside them (ol, oh)
    float il, ih, ol, oh;
    bool second;
};

// Runs of one direction from its prefix counts, and its gather windows.  Windows are symmetric about an integer
// bucket: a median run of an even number of buckets takes one more above.
//
// D_P: let ss be the smallest s with more than k2 keys in the buckets [ba - s, bb + s], w = bb - ba + 1.  A bucket b
// holds the keys of scaled value within 1/2 of b and the median m lies in the median run, so at least one MAD
// rank's deviation is not below ss - 1 and none is above ss + w bucket widths: the keys that hold those ranks lie
// within w + 1 buckets of bb + ss or of ba - ss.  The keys left out between the runs and outside them are bounded by
// the runs' edges, which sel_picks compares with the deviations it picks.
__device__ __forceinline__ SelRuns sel_runs(const unsigned* H, int nb, int n, bool ap, SelPar& par)
{
    const int lane = threadIdx.x & 31;
    const int k1 = (n - 1) / 2, k2 = n / 2, cap1 = (nb - NB2) / 2;
    auto P = [&](int b) { return b < 0 ? 0 : (int)H[b]; };
    SelRuns R{};
    const int ba = sel_find(H, nb, (unsigned)k1);
    int bb = k2 == k1 ? ba : sel_find(H, nb, (unsigned)k2);
    bb += (ba + bb) & 1;
    par.w0 = par.w1 = -1.0f;
    par.dd = 0.0f;
    par.nrc2 = 0ull;
    R.fb = 1;
    if (ba < 1 || bb > nb - 2) return R;   // an edge bucket holds every key beyond the range
    R.c_lo0 = P(ba - 1);
    R.cnt = R.cnt0 = P(bb) - R.c_lo0;
    if (R.cnt0 > sel_cap0(nb) || R.cnt0 > cap1) return R;
    R.fb = 0;
    const int mid = (ba + bb) / 2;
    par.nrc2 = dup2(-(TWO23 + (float)mid));
    par.w0 = R.wm = (float)(bb - mid);
    if (ap) {
        const int npos = (n & 1) ? (n - 1) / 2 : n / 2;   // keys above the median if none ties it
        if (npos > 0) {
            const int gb = n - npos;
            const int b3 = sel_find(H, nb, (unsigned)(gb + (npos - 1) / 2));
            int b4 = (npos & 1) ? b3 : sel_find(H, nb, (unsigned)(gb + npos / 2));
            if (b3 <= bb) {   // the runs meet: one window around both
                const int hw = max(b4, bb) - mid, lo = mid - hw, hi = mid + hw;
                if (lo >= 1 && hi <= nb - 2) {
                    const int below = P(lo - 1);
                    R.second = P(hi) - below <= cap1;
                    if (R.second) {
                        R.cnt = P(hi) - below;
                        R.c2 = below;
                        par.w0 = (float)hw;
                    }
                }
            } else {
                b4 += (b3 + b4) & 1;
                if (b4 <= nb - 2) {
                    const int c1 = P(b4) - P(b3 - 1);
                    R.second = c1 + R.cnt0 <= cap1;
                    if (R.second) {
                        R.cnt = c1 + R.cnt0;
                        R.c2 = P(b3 - 1) - R.cnt0;   // the listed keys below the run are the median run's
                        par.dd = (float)((b3 + b4) / 2 - mid);
                        par.w1 = (float)(b4 - (b3 + b4) / 2);
                    }
                }
            }
        }
        return R;
    }
    // the window count grows with s and reaches n: two levels of 32 lanes
    auto win = [&](int s) { return P(min(bb + s, nb - 1)) - P(ba - s - 1); };
    const int Q = nb >> 5;
    const int blk = __popc(__ballot_sync(0xFFFFFFFFu, win((lane + 1) * Q - 1) <= k2));
    int ss = blk * Q;
    for (int j = 0; j < Q; j += 32)
        ss += __popc(__ballot_sync(0xFFFFFFFFu, j + lane < Q && win(blk * Q + j + lane) <= k2));
    const int hw = bb - ba + 2;
    const int L0 = ba - ss - hw, L1 = ba - ss + hw, R0 = bb + ss - hw, R1 = bb + ss + hw;
    if (L0 >= 1 && R1 <= nb - 2) {
        const bool apart = L1 < ba;
        const int all = P(R1) - P(L0 - 1), left_out = apart ? (P(R0 - 1) - P(L1)) - R.cnt0 : 0;
        if (all - left_out <= cap1) {
            R.second = true;
            R.cnt = all - left_out;
            R.c2 = left_out;
            if (apart) {
                par.dd = (float)(bb + ss - mid);
                par.w1 = (float)hw;
            } else {
                par.w0 = (float)(R1 - mid);
            }
            // y of a scaled value v: (v - (of - 2^23)) / sc, a few roundings off: widened by 16 ulp
            const float o = par.of - TWO23, inv = __fdiv_rn(1.0f, par.sc);
            auto edge = [&](float v, float dir) {
                const float a = (v - o) * inv;
                return a + dir * 2e-6f * (fabsf(a) + fabsf(o * inv) + fabsf(v * inv));
            };
            R.il = edge((float)L1 + 0.5f, -1.0f);
            R.ih = edge((float)R0 - 0.5f, 1.0f);
            R.ol = edge((float)L0 - 0.5f, 1.0f);
            R.oh = edge((float)R1 + 0.5f, -1.0f);
        }
    }
    if (!R.second) R.fb = 2;
    return R;
}

// Lists one key.
__device__ __forceinline__ void sel_put(int* fill, float* B, int* I, int cap, float v, int i)
{
    const int pos = atomicAdd(fill, 1);
    if (pos < cap) {
        B[pos] = v;
        I[pos] = i;
    }
}

// Gather test of the keys y0 = (y_i, y_{i+1}), y1 = (y_{i+2}, y_{i+3}) of one direction; live: how many of them
// exist.  Raw bucket values are integers in [2^23, 2^24) inside the range, so r - rc is exact.
template <bool AP, bool TAIL>
__device__ __forceinline__ void sel_test(const SelPar& p, unsigned long long y0, unsigned long long y1, int i, int live,
                                         int* fill, float* B, int* I, int cap)
{
    const unsigned long long t0 = add2(fma2(y0, p.sc2, p.of2), p.nrc2), t1 = add2(fma2(y1, p.sc2, p.of2), p.nrc2);
    const float t[4] = {lo_f(t0), hi_f(t0), lo_f(t1), hi_f(t1)};
    bool h[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float a = (AP ? t[k] : fabsf(t[k])) - p.dd;
        h[k] = (fabsf(t[k]) <= p.w0) | (fabsf(a) <= p.w1);
        if (TAIL) h[k] = h[k] & (k < live);
    }
    if (h[0] | h[1] | h[2] | h[3]) {
        if (h[0]) sel_put(fill, B, I, cap, lo_f(y0), i);
        if (h[1]) sel_put(fill, B, I, cap, hi_f(y0), i + 1);
        if (h[2]) sel_put(fill, B, I, cap, lo_f(y1), i + 2);
        if (h[3]) sel_put(fill, B, I, cap, hi_f(y1), i + 3);
    }
}

// Exact selection of one rank over a direction's values f(0 .. L-1), all in [lo, hi], by iterated bucketing (the
// fallback): the value and the point index.  Each round keeps the rank's bucket and narrows [lo, hi] to the values
// in it, which lie in different buckets of the next round, so it ends.  Ranks are by value and then by point index;
// a group of more than 768 equal values (of more than 256 when all values are equal) gives its smallest index, as
// k_pdap2 does.
template <int GS, class CT, class F>
__device__ __noinline__ void sel_rank(const Grp<GS>& q, F f, int L, int rank, float lo, float hi, unsigned* H, float* TB,
                                      int* TI, CT& C, float& v, int& iv, int* err)
{
    // every histogram has at least this many words (a group of 512 threads takes nb >= 2,048)
    constexpr int FBN = GS > 256 ? 2048 : 1024, TCAP = 128, TIES = 768;
    int r = rank;
    for (int iter = 0; iter < 64; ++iter) {
        if (q.t == 0) {
            C.gn[q.g] = 0;
            C.gi[q.g] = 0x7FFFFFFF;
        }
        if (!(lo < hi)) {
            q.sync();
#pragma unroll 4
            for (unsigned i = q.t; i < (unsigned)L; i += GS)
                if (f((int)i) == lo) {
                    const int pos = atomicAdd(&C.gn[q.g], 1);
                    if (pos < TIES) H[pos] = i;
                    atomicMin(&C.gi[q.g], (int)i);
                }
            q.sync();
            const int T = C.gn[q.g];
            iv = T > 0 ? C.gi[q.g] : -1;   // values that are not numbers equal nothing
            v = lo;
            if (T > 0 && T <= (iter == 0 ? 256 : TIES)) {
                for (int t = q.t; t < T; t += GS) {
                    int below = 0;
                    for (int s = 0; s < T; ++s) below += H[s] < H[t];
                    if (below == r) C.pi1[q.g] = (int)H[t];
                }
                q.sync();
                iv = C.pi1[q.g];
            }
            q.sync();
            return;
        }
        float scale = __fdiv_rn((float)FBN, __fsub_rn(hi, lo));
        if (!(scale <= FLT_MAX)) scale = FLT_MAX;
        for (int b = q.t; b < FBN / 4; b += GS) reinterpret_cast<uint4*>(H)[b] = make_uint4(0u, 0u, 0u, 0u);
        q.sync();
#pragma unroll 4
        for (unsigned i = q.t; i < (unsigned)L; i += GS) {
            const float a = f((int)i);
            if (a >= lo && a <= hi) atomicAdd(&H[bucket<FBN>(a, lo, scale)], 1u);
        }
        q.sync();
        int b1, c1, b2, c2;
        gfind<GS, CT, FBN>(q, H, r, r, C, b1, c1, b2, c2);
        const int cnt = (int)H[b1];
        r -= c1;
        if (cnt <= TCAP) {
#pragma unroll 4
            for (unsigned i = q.t; i < (unsigned)L; i += GS) {
                const float a = f((int)i);
                if (a >= lo && a <= hi && bucket<FBN>(a, lo, scale) == b1) {
                    const int pos = atomicAdd(&C.gn[q.g], 1);
                    if (pos < TCAP) {
                        TB[pos] = a;
                        TI[pos] = (int)i;
                    }
                }
            }
            q.sync();
            float v2;
            int i2;
            gpick(q, TB, TI, cnt, r, r, C, v, v2, iv, i2);
            return;
        }
        float nlo = FLT_MAX, nhi = -FLT_MAX;
#pragma unroll 4
        for (unsigned i = q.t; i < (unsigned)L; i += GS) {
            const float a = f((int)i);
            if (a >= lo && a <= hi && bucket<FBN>(a, lo, scale) == b1) {
                nlo = fminf(nlo, a);
                nhi = fmaxf(nhi, a);
            }
        }
        gminmax(q, nlo, nhi, C, lo, hi);
    }
    if (q.t == 0) atomicOr(err, ERR_SELECT_ITER);
    v = __int_as_float(0x7FC00000);
    iv = -1;
}

// Two ranks s1 <= s2 by sel_rank.
template <int GS, class CT, class F>
__device__ __forceinline__ void sel_ranks(const Grp<GS>& q, F f, int L, int s1, int s2, float lo, float hi, unsigned* H,
                                          float* TB, int* TI, CT& C, float& v1, float& v2, int& i1, int& i2, int* err)
{
    sel_rank<GS, CT, F>(q, f, L, s1, lo, hi, H, TB, TI, C, v1, i1, err);
    v2 = v1;
    i2 = i1;
    if (s2 != s1) sel_rank<GS, CT, F>(q, f, L, s2, lo, hi, H, TB, TI, C, v2, i2, err);
}

// The warp form of the picks, for lists of up to 32 FJ keys with at most 32 in the median run: the list sits in
// registers, small sets are ranked by shuffles (independent of each other, where a loop over shared memory waits
// for each load), and a larger one is first cut down by a 32-bin histogram.
constexpr int FJ = 8;

// Ranks s1 <= s2 (by value, then point index) among the cnt <= 32 pairs held one per lane.
__device__ __forceinline__ void warp_rank(float v, int iv, int cnt, int s1, int s2, float& v1, float& v2, int& i1, int& i2)
{
    const int lane = threadIdx.x & 31;
    int r = 0;
    for (int s = 0; s < cnt; ++s) {
        const float o = __shfl_sync(0xFFFFFFFFu, v, s);
        const int oi = __shfl_sync(0xFFFFFFFFu, iv, s);
        r += (o < v) | ((o == v) & (oi < iv));
    }
    const unsigned m1 = __ballot_sync(0xFFFFFFFFu, lane < cnt && r == s1);
    const unsigned m2 = __ballot_sync(0xFFFFFFFFu, lane < cnt && r == s2);
    const int l1 = __ffs(m1) - 1, l2 = __ffs(m2) - 1;
    v1 = __shfl_sync(0xFFFFFFFFu, v, l1 < 0 ? 0 : l1);
    i1 = __shfl_sync(0xFFFFFFFFu, iv, l1 < 0 ? 0 : l1);
    v2 = __shfl_sync(0xFFFFFFFFu, v, l2 < 0 ? 0 : l2);
    i2 = __shfl_sync(0xFFFFFFFFu, iv, l2 < 0 ? 0 : l2);
}

// Moves the kept of the warp's pairs (bit j of keep: pair j of this lane) to (TB, TI), at most 32; their number.
__device__ __forceinline__ int warp_pack(const float (&v)[FJ], const int (&iv)[FJ], unsigned keep, int nj, float* TB, int* TI)
{
    const int lane = threadIdx.x & 31;
    int base = 0;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < FJ; ++j)
        if (j < nj) {
            const bool k = (keep >> j) & 1u;
            const unsigned m = __ballot_sync(0xFFFFFFFFu, k);
            const int pos = base + __popc(m & ((1u << lane) - 1u));
            if (k && pos < 32) {
                TB[pos] = v[j];
                TI[pos] = iv[j];
            }
            base += __popc(m);
        }
    __syncwarp();
    return base;
}

// Ranks s1 <= s2 among the warp's cnt pairs; [lo, hi]: where the values of interest lie (any bins would do).  False
// when more than 32 pairs share the ranks' bins.
__device__ __forceinline__ bool warp_select(const float (&v)[FJ], const int (&iv)[FJ], int cnt, int s1, int s2, float lo,
                                            float hi, unsigned* bins, float* TB, int* TI, float& v1, float& v2, int& i1,
                                            int& i2)
{
    const int lane = threadIdx.x & 31, nj = (cnt + 31) >> 5;
    const float sc = hi > lo ? __fdiv_rn(32.0f, __fsub_rn(hi, lo)) : 0.0f;   // no range: one bin
    int b[FJ];
    bins[lane] = 0u;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < FJ; ++j)
        if (j < nj) {
            b[j] = __float2int_rz(fminf(fmaxf(__fmul_rn(__fsub_rn(v[j], lo), sc), 0.0f), 31.0f));
            if (j * 32 + lane < cnt) atomicAdd(&bins[b[j]], 1u);
        }
    __syncwarp();
    int incl = (int)bins[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    const int b1 = __popc(__ballot_sync(0xFFFFFFFFu, incl <= s1)), b2 = __popc(__ballot_sync(0xFFFFFFFFu, incl <= s2));
    if (b2 > 31) return false;
    const int below = b1 ? __shfl_sync(0xFFFFFFFFu, incl, b1 - 1) : 0;
    const int n2 = __shfl_sync(0xFFFFFFFFu, incl, b2) - below;
    if (n2 > 32) return false;
    unsigned keep = 0;
#pragma unroll
    for (int j = 0; j < FJ; ++j)
        if (j < nj) keep |= (unsigned)(j * 32 + lane < cnt && b[j] >= b1 && b[j] <= b2) << j;
    warp_pack(v, iv, keep, nj, TB, TI);
    warp_rank(TB[lane], TI[lane], n2, s1 - below, s2 - below, v1, v2, i1, i2);
    return true;
}

// The picks of one direction by one warp (see sel_picks, whose steps these are); false where sel_picks must decide.
__device__ __forceinline__ bool sel_picks_warp(const SelRuns& R, const SelPar& par, unsigned* H, int nb, int n, bool ap,
                                               ResDev* out)
{
    const int lane = threadIdx.x & 31, nj = (R.cnt + 31) >> 5;
    const int k1 = (n - 1) / 2, k2 = n / 2, cap0 = sel_cap0(nb), cap1 = (nb - NB2) / 2;
    float* TB = reinterpret_cast<float*>(H + nb);
    int* TI = reinterpret_cast<int*>(TB + cap0);
    const float* B = reinterpret_cast<const float*>(H + NB2);
    const int* I = reinterpret_cast<const int*>(H + NB2 + cap1);
    float v[FJ];
    int iv[FJ];
    unsigned keep = 0;
    const float nrc = lo_f(par.nrc2);
#pragma unroll
    for (int j = 0; j < FJ; ++j)
        if (j < nj) {
            const bool in = j * 32 + lane < R.cnt;
            v[j] = in ? B[j * 32 + lane] : 0.0f;
            iv[j] = in ? I[j * 32 + lane] : 0;
            keep |= (unsigned)(in && fabsf(__fadd_rn(__fmaf_rn(v[j], par.sc, par.of), nrc)) <= R.wm) << j;
        }
    warp_pack(v, iv, keep, nj, TB, TI);
    float m1, m2, p1, p2;
    int im1, im2, ip1 = NOPOS, ip2 = NOPOS;
    const float tv = TB[lane];
    warp_rank(tv, TI[lane], R.cnt0, k1 - R.c_lo0, k2 - R.c_lo0, m1, m2, im1, im2);
    if (ap) {
        const int nle = R.c_lo0 + __popc(__ballot_sync(0xFFFFFFFFu, lane < R.cnt0 && tv <= m1));
        const int npos = n - nle;
        if (npos > 0) {
            const int s3 = nle + (npos - 1) / 2 - R.c2, s4 = nle + npos / 2 - R.c2;
            if (!R.second || s3 < (par.w1 < 0.0f ? 0 : R.cnt0) || s4 >= R.cnt) return false;
            // the second window's edges (or the whole window's), about
            const float o = -nrc - par.of, inv = __fdiv_rn(1.0f, par.sc);
            const float lo = (o + (par.w1 < 0.0f ? -par.w0 : par.dd - par.w1) - 0.5f) * inv;
            const float hi = (o + (par.w1 < 0.0f ? par.w0 : par.dd + par.w1) + 0.5f) * inv;
            if (!warp_select(v, iv, R.cnt, s3, s4, lo, hi, H, TB, TI, p1, p2, ip1, ip2)) return false;
        }
    } else {
        const float m = __fmul_rn(__fadd_rn(m1, m2), 0.5f);
        const float inner = R.c2 ? fmaxf(__fsub_rn(m, R.il), __fsub_rn(R.ih, m)) : -1.0f;
        const float outer = fminf(__fsub_rn(m, R.ol), __fsub_rn(R.oh, m));
        const int s1 = k1 - R.c2, s2 = k2 - R.c2;
        if (s1 < 0 || s2 >= R.cnt || !(inner < outer)) return false;
#pragma unroll
        for (int j = 0; j < FJ; ++j)
            if (j < nj) v[j] = fabsf(__fsub_rn(v[j], m));
        if (!warp_select(v, iv, R.cnt, s1, s2, fmaxf(inner, 0.0f), outer, H, TB, TI, p1, p2, ip1, ip2)) return false;
        if (!(inner < p1 && outer > p2)) return false;
    }
    if (lane == 0) put_picks(out, im1, im2, ip1, ip2);
    return true;
}

// The picks of one direction from its list, the iterated selection where that failed, and the result cell.
// y.get(i): key of point i.  H: the direction's sel_words(nb) words, the list after NB2 words.
template <int GS, class CT, class K>
__device__ __noinline__ void sel_picks(const Grp<GS> q, const K y, const SelRuns R, const SelPar par, CT& C,
                                       unsigned* H, int nb, int n, bool ap, ResDev* out, int* err)
{
    constexpr int TCAP = 128;
    const int k1 = (n - 1) / 2, k2 = n / 2, cap0 = sel_cap0(nb), cap1 = (nb - NB2) / 2;
    float* TB = reinterpret_cast<float*>(H + nb);
    int* TI = reinterpret_cast<int*>(TB + cap0);
    float* B = reinterpret_cast<float*>(H + NB2);
    int* I = reinterpret_cast<int*>(H + NB2 + cap1);
    const float qnan = __int_as_float(0x7FC00000);
    float m1 = qnan, m2 = qnan, p1 = 0.f, p2 = 0.f;
    int im1 = -1, im2 = -1, ip1 = -1, ip2 = -1, npos = 0, fb = R.fb;
    // the list must hold the keys the counts promise
    if (fb != 1 && C.fill[q.g][0] != R.cnt) fb = 1;
    if (fb != 1) {
        // the median run's keys, listed apart
        if (q.t == 0) C.fill[q.g][1] = 0;
        q.sync();
        const float nrc = lo_f(par.nrc2);
        for (int t = q.t; t < R.cnt; t += GS) {
            const float v = B[t];
            if (fabsf(__fadd_rn(__fmaf_rn(v, par.sc, par.of), nrc)) <= R.wm)
                sel_put(&C.fill[q.g][1], TB, TI, cap0, v, I[t]);
        }
        q.sync();
        gpick(q, TB, TI, R.cnt0, k1 - R.c_lo0, k2 - R.c_lo0, C, m1, m2, im1, im2);
        if (ap) {
            // #(y <= med) = #(y <= m1): keys below the run plus its keys <= m1
            int c = 0;
            for (int t = q.t; t < R.cnt0; t += GS) c += (TB[t] <= m1);
            const int nle = R.c_lo0 + gsum(q, c, C);
            npos = n - nle;
            if (npos > 0) {
                const int s3 = nle + (npos - 1) / 2 - R.c2, s4 = nle + npos / 2 - R.c2;
                // the listed keys of the second run are the list's last ones in rank
                if (!R.second || s3 < (par.w1 < 0.0f ? 0 : R.cnt0) || s4 >= R.cnt) {
                    fb = 2;   // no run, or the positive count differed from the guess
                } else if (R.cnt <= 64) {
                    gpick(q, B, I, R.cnt, s3, s4, C, p1, p2, ip1, ip2);
                } else {
                    float lo = FLT_MAX, hi = -FLT_MAX;
                    for (int t = q.t; t < R.cnt; t += GS) {
                        lo = fminf(lo, B[t]);
                        hi = fmaxf(hi, B[t]);
                    }
                    gminmax(q, lo, hi, C, lo, hi);
                    gpick_wide<GS, CT, TCAP>(q, B, I, R.cnt, s3, s4, lo, hi, H, TB, TI, C, p1, p2, ip1, ip2);
                }
            }
        } else if (fb == 0) {
            const float m = __fmul_rn(__fadd_rn(m1, m2), 0.5f);
            for (int t = q.t; t < R.cnt; t += GS) B[t] = fabsf(__fsub_rn(B[t], m));
            q.sync();
            // deviations of the keys left out: at most inner between the runs, at least outer outside them
            const float inner = R.c2 ? fmaxf(__fsub_rn(m, R.il), __fsub_rn(R.ih, m)) : -1.0f;
            const float outer = fminf(__fsub_rn(m, R.ol), __fsub_rn(R.oh, m));
            const int s1 = k1 - R.c2, s2 = k2 - R.c2;
            if (s1 < 0 || s2 >= R.cnt || !(inner < outer)) {
                fb = 2;
            } else {
                // picks within [inner, outer], or the direction falls back: a histogram over that range serves
                gpick_wide<GS, CT, TCAP>(q, B, I, R.cnt, s1, s2, fmaxf(inner, 0.0f), outer, H, TB, TI, C, p1, p2, ip1,
                                         ip2);
                if (!(inner < p1 && outer > p2)) fb = 2;   // strictly: no key left out ties a pick
            }
        }
    }
    if (fb) {
        q.sync();
        auto f = [&](int i) { return y.get(i); };
        float kl = FLT_MAX, kh = -FLT_MAX;
#pragma unroll 4
        for (unsigned i = q.t; i < (unsigned)n; i += GS) {
            const float v = y.get(i);
            kl = fminf(kl, v);
            kh = fmaxf(kh, v);
        }
        gminmax(q, kl, kh, C, kl, kh);
        if (fb == 1)
            sel_ranks(q, f, n, k1, k2, kl, kh, H, TB, TI, C, m1, m2, im1, im2, err);
        if (ap) {
            int c = 0;
            for (unsigned i = q.t; i < (unsigned)n; i += GS) c += (y.get(i) <= m1);
            const int nle = gsum(q, c, C);
            npos = n - nle;
            ip1 = ip2 = -1;
            if (npos > 0)
                sel_ranks(q, f, n, nle + (npos - 1) / 2, nle + npos / 2, kl, kh, H, TB, TI, C, p1, p2, ip1, ip2, err);
        } else {
            const float m = __fmul_rn(__fadd_rn(m1, m2), 0.5f);
            const float dmax = fmaxf(fabsf(__fsub_rn(kl, m)), fabsf(__fsub_rn(kh, m)));
            auto fd = [&](int i) { return fabsf(__fsub_rn(y.get(i), m)); };
            sel_ranks(q, fd, n, k1, k2, 0.0f, dmax, H, TB, TI, C, p1, p2, ip1, ip2, err);
        }
    }
    if (q.t == 0) put_picks(out, im1, im2, ap && npos == 0 ? NOPOS : ip1, ap && npos == 0 ? NOPOS : ip2);
}

// Counts a key of raw bucket value r; hb: shared address of the histogram minus 4 MAGIC, so that the float's bits
// are the index.
__device__ __forceinline__ void sel_count(unsigned hb, int top, float r)
{
    const int b = min(max(__float_as_int(r), MAGIC), top);
    // no memory clobber: the barriers on either side of a pass order it, and loads may move across it
    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(hb + 4u * (unsigned)b));
}
__device__ __forceinline__ unsigned sel_base(const unsigned* H)
{
    return (unsigned)__cvta_generic_to_shared(H) - 4u * (unsigned)MAGIC;
}

// Keys in device memory (kin: G x npad per task in launch order, formed by launch_pdap_keys): one block of GS
// threads per direction, so directions never wait for one another and a block's few barriers are its own.
// Bound by the shared-memory reductions and the issue slots of the two passes, about 14 instructions per key.
template <int GS>
__global__ void __launch_bounds__(GS, 1024 / GS) k_select(const TaskDev* __restrict__ tasks, int G,
                                               const SlotDev* __restrict__ slots, const DsDev* __restrict__ dsets,
                                               ResDev* __restrict__ res, int* err, const float* __restrict__ kin, int nb)
{
    extern __shared__ __align__(16) unsigned sel_sm[];
    __shared__ CtlS<1> C;
    const int ti = blockIdx.x / G, g = blockIdx.x - ti * G;
    const TaskDev T = tasks[ti];
    if (g >= T.nj) return;
    const SlotDev& S = slots[T.slot];
    const int n = (int)dsets[T.ds].n, npad = (n + 3) & ~3;
    const float rad = dsets[T.ds].rc;
    const bool ap = S.kind == 2;
    unsigned* H = sel_sm;   // sel_words(nb) words
    const KeysArray y{kin + (size_t)blockIdx.x * npad};
    const Grp<GS> q{0, (int)threadIdx.x};
    const int lane = q.t & 31;
    for (int b = q.t; b < nb / 4; b += GS) reinterpret_cast<uint4*>(H)[b] = make_uint4(0u, 0u, 0u, 0u);
    if (q.t < 2) C.fill[0][q.t] = 0;
    SelPar par{};
    float sample[RS];
#pragma unroll
    for (int k = 0; k < RS; ++k) sample[k] = y.y[sel_sample(n, lane, k)];
    sel_range(sample, rad, nb, par);   // every warp for itself: the same values
    q.sync();
    // copies for the passes: par itself goes to calls by reference and so lives in local memory
    const unsigned long long sc2 = par.sc2, of2 = par.of2;

    const unsigned n4 = (unsigned)n & ~3u, STEP = 4 * GS;   // unsigned: n may be close to 2^31
    const unsigned hb = sel_base(H);
    const int top = MAGIC + nb - 1;
    auto load = [&](unsigned i) { return *reinterpret_cast<const ulonglong2*>(y.y + i); };
    auto count4 = [&](const ulonglong2& v) {
        const unsigned long long r0 = fma2(v.x, sc2, of2), r1 = fma2(v.y, sc2, of2);
        sel_count(hb, top, lo_f(r0));
        sel_count(hb, top, hi_f(r0));
        sel_count(hb, top, lo_f(r1));
        sel_count(hb, top, hi_f(r1));
    };
    unsigned i = 4 * q.t;
    for (; i + 3 * STEP < n4; i += 4 * STEP) {
        const ulonglong2 a = load(i), b = load(i + STEP), c = load(i + 2 * STEP), d = load(i + 3 * STEP);
        count4(a);
        count4(b);
        count4(c);
        count4(d);
    }
    for (; i < n4; i += STEP) count4(load(i));
    if (n4 + q.t < (unsigned)n) sel_count(hb, top, __fmaf_rn(y.get(n4 + q.t), par.sc, par.of));
    q.sync();

    sel_prefix(q, H, nb, C);
    const SelRuns R = sel_runs(H, nb, n, ap, par);
    q.sync();   // the histogram's memory takes the list from here
    if (R.fb != 1) {
        const SelPar pg = par;
        const int cap1 = (nb - NB2) / 2;
        float* B = reinterpret_cast<float*>(H + NB2);
        int* I = reinterpret_cast<int*>(H + NB2 + cap1);
        auto gather = [&](auto apc) {
            constexpr bool AP = decltype(apc)::value;
            auto test4 = [&](const ulonglong2& v, unsigned at) {
                sel_test<AP, false>(pg, v.x, v.y, (int)at, 4, &C.fill[0][0], B, I, cap1);
            };
            unsigned i = 4 * q.t;
            for (; i + 3 * STEP < n4; i += 4 * STEP) {
                const ulonglong2 a = load(i), b = load(i + STEP), c = load(i + 2 * STEP), d = load(i + 3 * STEP);
                test4(a, i);
                test4(b, i + STEP);
                test4(c, i + 2 * STEP);
                test4(d, i + 3 * STEP);
            }
            for (; i < n4; i += STEP) test4(load(i), i);
            if (i < (unsigned)n) {   // the last, partial four (the row is padded to whole fours)
                const ulonglong2 v = load(i);
                sel_test<AP, true>(pg, v.x, v.y, (int)i, n - (int)i, &C.fill[0][0], B, I, cap1);
            }
        };
        if (ap) gather(TrueT{});
        else gather(FalseT{});
        q.sync();
    }
    ResDev* out = res + S.roff + T.j0 + g;
    if (R.fb == 0 && R.cnt <= 32 * FJ && R.cnt0 <= 32 && C.fill[0][0] == R.cnt) {   // the same in every thread
        if (q.t < 32) {
            const bool ok = sel_picks_warp(R, par, H, nb, n, ap, out);
            if (q.t == 0) C.gi[0] = ok;
        }
        q.sync();
        if (C.gi[0]) return;
        q.sync();
    }
    sel_picks<GS, CtlS<1>, KeysArray>(q, y, R, par, C, H, nb, n, ap, out, err);
}

// A key is two half chains over the dims, added (key_halves), here without the zero-padded terms (a zero product
// leaves a chain unchanged): the values the other selection kernels form.
template <int D>
struct HalfChains {
    static constexpr int DP4 = (D + 3) & ~3, H2 = DP4 / 2, E0 = D < H2 ? D : H2;
};

// One direction's keys re-formed one by one, for the range sample and the iterated selection (any d <= 16; u: the
// direction's pairs (u, u) in shared memory).
struct KeysFromX {
    const float* X;
    const float2* u;
    int ldx, d;
    __device__ __forceinline__ float get(int i) const
    {
        const float4* x = reinterpret_cast<const float4*>(X + (int64_t)i * ldx);
        const int nc = (d + 3) >> 2, h2 = 2 * nc;
        float4 xv[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) xv[c] = c < nc ? x[c] : make_float4(0.f, 0.f, 0.f, 0.f);
        float p0 = 0.f, p1 = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float e[4] = {xv[c].x, xv[c].y, xv[c].z, xv[c].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int l = 4 * c + k;
                if (l < d) {
                    if (l < h2) p0 = fmaf(u[l].x, e[k], p0);
                    else p1 = fmaf(u[l].x, e[k], p1);
                }
            }
        }
        return __fadd_rn(p0, p1);
    }
};

// Points per thread of k_select_x: NG groups of four consecutive points, 128 points apart, so that a warp takes chunks
// of 128 NG points whose loads lie side by side.  Two groups where their coordinates fit the registers.
template <int D>
struct PointGroups {
    static constexpr int NG = D <= 11 ? 2 : 1, CHUNK = 128 * NG;
};

// The four points i .. i + 3 as pairs: x[l][0] = (x_i[l], x_{i+1}[l]), x[l][1] the next two.  From the dataset's
// columns (Xt: dim l of point i at l * colst + i, zero beyond n up to a multiple of 32) or, without them, from the
// padded rows (points beyond n repeat the last one).  i < n.
template <int D, int S>
__device__ __forceinline__ void load_points(const DsDev& Dd, unsigned i, int n, unsigned long long (&xv)[D][S], int at)
{
    if (Dd.Xt) {
        const size_t colst = (size_t)((n + 31) & ~31);
#pragma unroll
        for (int l = 0; l < D; ++l) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(Dd.Xt + l * colst + i);
            xv[l][at] = v.x;
            xv[l][at + 1] = v.y;
        }
        return;
    }
    constexpr int D4 = (D + 3) & ~3;
    float x[4][D4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4* xr = reinterpret_cast<const float4*>(Dd.X32 + (int64_t)min(i + k, (unsigned)n - 1u) * Dd.ldx);
#pragma unroll
        for (int c = 0; c < D4 / 4; ++c) {
            const float4 t4 = xr[c];
            x[k][4 * c] = t4.x;
            x[k][4 * c + 1] = t4.y;
            x[k][4 * c + 2] = t4.z;
            x[k][4 * c + 3] = t4.w;
        }
    }
#pragma unroll
    for (int l = 0; l < D; ++l) {
        asm("mov.b64 %0, {%1, %2};" : "=l"(xv[l][at]) : "f"(x[0][l]), "f"(x[1][l]));
        asm("mov.b64 %0, {%1, %2};" : "=l"(xv[l][at + 1]) : "f"(x[2][l]), "f"(x[3][l]));
    }
}

// The keys of one direction (u: D pairs (u, u) in shared memory) for the thread's points, as pairs.
template <int D, int S>
__device__ __forceinline__ void form_keys(const float2* u, const unsigned long long (&xv)[D][S], unsigned long long (&k)[S])
{
    using HC = HalfChains<D>;
    unsigned long long p0[S], p1[S];
#pragma unroll
    for (int h = 0; h < S; ++h) p0[h] = p1[h] = 0ull;
#pragma unroll
    for (int l = 0; l < D; l += 2) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(u + l);   // padded to an even count
        const unsigned long long uu[2] = {v.x, v.y};
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (l + e < D) {
#pragma unroll
                for (int h = 0; h < S; ++h) {
                    if (l + e < HC::E0) p0[h] = fma2(uu[e], xv[l + e][h], p0[h]);
                    else p1[h] = fma2(uu[e], xv[l + e][h], p1[h]);
                }
            }
    }
#pragma unroll
    for (int h = 0; h < S; ++h) k[h] = HC::H2 < D ? add2(p0[h], p1[h]) : p0[h];
}

// d <= 16: keys re-formed from X at both passes.  The whole CTA walks the points, four per thread with their
// coordinates in registers, and forms their keys for every direction of the task (packed FMAs over point pairs,
// the direction's pairs from shared memory); warp g then takes direction g's steps between the passes alone.
// X is read twice per task whatever its number of directions, and no key is stored, so 16 directions are in flight
// per SM at any n.  About 25 instructions per key over both passes.
template <int D>
__global__ void __launch_bounds__(SX_NT, 2) k_select_x(const TaskDev* __restrict__ tasks,
                                                     const SlotDev* __restrict__ slots,
                                                     const DsDev* __restrict__ dsets, const float* __restrict__ U,
                                                     ResDev* __restrict__ res, int* err, int nb, int G)
{
    constexpr int DU = (D + 1) & ~1;
    extern __shared__ __align__(16) unsigned sel_sm[];
    __shared__ CtlS<SX_G> C;
    const TaskDev T = tasks[blockIdx.x];
    const SlotDev& S = slots[T.slot];
    const DsDev Dd = dsets[T.ds];
    const int n = (int)Dd.n, ldx = Dd.ldx, GA = T.nj, NT = blockDim.x;
    const bool ap = S.kind == 2;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int words = sel_words(nb);
    unsigned* area = sel_sm;                                              // G x words
    float2* uS = reinterpret_cast<float2*>(area + (size_t)G * words);     // G x DU pairs (u, u)
    const float* Ut = U + S.uoff + (int64_t)T.j0 * ldx;
    for (int e = tid; e < G * DU; e += NT) {
        const int g = e / DU, l = e - g * DU;
        const float u = (g < GA && l < D) ? Ut[(int64_t)g * ldx + l] : 0.0f;
        uS[e] = make_float2(u, u);
    }
    for (int g = 0; g < GA; ++g)
        for (int e = tid; e < nb / 4; e += NT) reinterpret_cast<uint4*>(area + g * words)[e] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    const Grp<32> q{w, lane};
    const KeysFromX y{Dd.X32, uS + w * DU, ldx, D};
    SelPar par{};
    if (w < GA) {
        float sample[RS];
#pragma unroll
        for (int k = 0; k < RS; ++k) sample[k] = y.get(sel_sample(n, lane, k));
        sel_range(sample, Dd.rc, nb, par);
        if (lane == 0) {
            C.par[w] = par;
            C.fill[w][0] = 0;
        }
    }
    __syncthreads();

    using PG = PointGroups<D>;
    constexpr int NG = PG::NG, S2 = 2 * NG;
    const unsigned hb0 = sel_base(area);
    const int top = MAGIC + nb - 1, nwarps = NT >> 5;
    // unsigned: n may be close to 2^31
    for (unsigned base = w * PG::CHUNK; base < (unsigned)n; base += nwarps * PG::CHUNK) {
        const unsigned i = base + 4 * lane;
        unsigned long long xv[D][S2] = {};
#pragma unroll
        for (int p = 0; p < NG; ++p)
            if (i + 128 * p < (unsigned)n) load_points<D, S2>(Dd, i + 128 * p, n, xv, 2 * p);
        if (base + PG::CHUNK <= (unsigned)n) {
#pragma unroll 1
            for (int g = 0; g < GA; ++g) {
                unsigned long long k[S2];
                form_keys<D, S2>(uS + g * DU, xv, k);
                const ulonglong2 so = *reinterpret_cast<const ulonglong2*>(&C.par[g].sc2);
                const unsigned hb = hb0 + 4u * (unsigned)(g * words);
#pragma unroll
                for (int h = 0; h < S2; ++h) {
                    const unsigned long long r = fma2(k[h], so.x, so.y);
                    sel_count(hb, top, lo_f(r));
                    sel_count(hb, top, hi_f(r));
                }
            }
        } else {
#pragma unroll 1
            for (int g = 0; g < GA; ++g) {
                unsigned long long k[S2];
                form_keys<D, S2>(uS + g * DU, xv, k);
                const ulonglong2 so = *reinterpret_cast<const ulonglong2*>(&C.par[g].sc2);
                const unsigned hb = hb0 + 4u * (unsigned)(g * words);
#pragma unroll
                for (int h = 0; h < S2; ++h) {
                    const unsigned long long r = fma2(k[h], so.x, so.y);
                    const unsigned at = i + 128 * (h >> 1) + 2 * (h & 1);
                    if (at < (unsigned)n) sel_count(hb, top, lo_f(r));
                    if (at + 1 < (unsigned)n) sel_count(hb, top, hi_f(r));
                }
            }
        }
    }
    __syncthreads();

    SelRuns R{};
    unsigned* H = area + w * words;
    if (w < GA) {
        sel_prefix(q, H, nb, C);
        R = sel_runs(H, nb, n, ap, par);
        if (lane == 0) C.par[w] = par;   // no window where the iterated selection takes the direction
    }
    __syncthreads();

    const int cap1 = (nb - NB2) / 2;
    auto gather = [&](auto apc) {
        constexpr bool AP = decltype(apc)::value;
        for (unsigned base = w * PG::CHUNK; base < (unsigned)n; base += nwarps * PG::CHUNK) {
            const unsigned i = base + 4 * lane;
            unsigned long long xv[D][S2] = {};
#pragma unroll
            for (int p = 0; p < NG; ++p)
                if (i + 128 * p < (unsigned)n) load_points<D, S2>(Dd, i + 128 * p, n, xv, 2 * p);
            int live[NG];   // points of each group that exist
#pragma unroll
            for (int p = 0; p < NG; ++p)
                live[p] = i + 128 * p < (unsigned)n ? (int)min(4u, (unsigned)n - (i + 128 * p)) : 0;
            auto dirs = [&](auto tailc) {
                constexpr bool TAIL = decltype(tailc)::value;
#pragma unroll 1
                for (int g = 0; g < GA; ++g) {
                    unsigned long long k[S2];
                    form_keys<D, S2>(uS + g * DU, xv, k);
                    const SelPar pg = C.par[g];
                    unsigned* L = area + g * words + NB2;
#pragma unroll
                    for (int p = 0; p < NG; ++p)
                        sel_test<AP, TAIL>(pg, k[2 * p], k[2 * p + 1], (int)(i + 128 * p), live[p], &C.fill[g][0], reinterpret_cast<float*>(L), reinterpret_cast<int*>(L + cap1),
                                           cap1);
                }
            };
            if (base + PG::CHUNK <= (unsigned)n) dirs(FalseT{});
            else dirs(TrueT{});
        }
    };
    if (ap) gather(TrueT{});
    else gather(FalseT{});
    __syncthreads();
    if (w >= GA) return;
    ResDev* out = res + S.roff + T.j0 + w;
    if (R.fb == 0 && R.cnt <= 32 * FJ && R.cnt0 <= 32 && C.fill[w][0] == R.cnt &&
        sel_picks_warp(R, par, H, nb, n, ap, out))
        return;
    sel_picks<32, CtlS<SX_G>, KeysFromX>(q, y, R, par, C, H, nb, n, ap, out, err);
}

// Buckets per direction by n: about 16 n / nb keys are listed for D_P and 0.001 x 2048 / nb x n lie in a bucket
// at the median (normal data), so these lines keep both well inside their buffers while the histograms stay small
// enough for 16 (k_select_x: nb = 2,048, 165 KB) or some 20 (k_select) directions per SM.
int sel_buckets(int64_t n)
{
    return n <= 4000 ? 1024 : (n <= 32000 ? 2048 : (n <= 130000 ? 4096 : 8192));
}

size_t sel_smem(int nb, int G, int d)
{
    return sizeof(unsigned) * (size_t)G * sel_words(nb) + (d ? sizeof(float2) * (size_t)G * ((d + 1) & ~1) : 0);
}

template <int D>
cudaError_t launch_x(const TaskDev* tasks, int ntasks, int G, int nb, const SlotDev* slots, const DsDev* ds,
                            const float* U, ResDev* res, int* err, cudaStream_t st)
{
    const size_t smem = sel_smem(nb, G, D);
    static SmemLimit limit;
    const cudaError_t e = limit.raise(k_select_x<D>);
    if (e != cudaSuccess) return e;
    k_select_x<D><<<ntasks, SX_NT, smem, st>>>(tasks, slots, ds, U, res, err, nb, G);
    return cudaGetLastError();
}

template <int GS>
cudaError_t launch_k(const TaskDev* tasks, int ntasks, int G, int nb, const SlotDev* slots, const DsDev* ds,
                            ResDev* res, int* err, const float* kin, cudaStream_t st)
{
    const size_t smem = sel_smem(nb, 1, 0);
    static SmemLimit limit;
    const cudaError_t e = limit.raise(k_select<GS>);
    if (e != cudaSuccess) return e;
    k_select<GS><<<ntasks * G, GS, smem, st>>>(tasks, G, slots, ds, res, err, kin, nb);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sel(const TaskDev* tasks, int ntasks, int group, int variant, const SlotDev* slots, const DsDev* ds,
                       const float* U, ResDev* res, int* err, cudaStream_t st, const float* kin)
{
    if (variant & PDAP_WARP) {
        const int d = variant & 0xFF, nb = 1 << ((variant >> 16) & 31);
        if (group < 1 || group > SX_G) return cudaErrorInvalidValue;
#define RRS_X(D) \
    case D: return launch_x<D>(tasks, ntasks, group, nb, slots, ds, U, res, err, st);
        switch (d) {
            RRS_X(1) RRS_X(2) RRS_X(3) RRS_X(4) RRS_X(5) RRS_X(6) RRS_X(7) RRS_X(8)
            RRS_X(9) RRS_X(10) RRS_X(11) RRS_X(12) RRS_X(13) RRS_X(14) RRS_X(15) RRS_X(16)
        default: return cudaErrorInvalidValue;
        }
#undef RRS_X
    }
    {
        if (!kin) return cudaErrorInvalidValue;
        // one warp per direction for short arrays, more where one warp's pass would be long or where the launch has
        // too few directions to give every SM some 48 warps (its loads are what the passes wait for)
        const int nb = 1 << ((variant >> 16) & 31);
        const int64_t dirs = (int64_t)ntasks * group;
        int gs = nb > 4096 ? 256 : (nb > 2048 ? 128 : (nb > 1024 ? 64 : 32));
        while (gs < 512 && dirs * gs < 152 * 32 * 48 && gs * 16 < nb * 4) gs *= 2;
        switch (gs) {
        case 32: return launch_k<32>(tasks, ntasks, group, nb, slots, ds, res, err, kin, st);
        case 64: return launch_k<64>(tasks, ntasks, group, nb, slots, ds, res, err, kin, st);
        case 128: return launch_k<128>(tasks, ntasks, group, nb, slots, ds, res, err, kin, st);
        case 256: return launch_k<256>(tasks, ntasks, group, nb, slots, ds, res, err, kin, st);
        default: return launch_k<512>(tasks, ntasks, group, nb, slots, ds, res, err, kin, st);
        }
    }
}

PdapShape pdap_shape(int n, int ldx, int m, int d, int group, int64_t rows)
{
    PdapShape s{};
    const int dp4 = pdap_dp4_class(d), nb = sel_buckets(n);
    int lg = 0;
    while ((1 << lg) < nb) ++lg;
    if (group == 1 || group == 2 || group == 4) {
        // asked for: that many directions per CTA with resident keys, where they fit
        if (group <= m && pdap_smem_bytes(n, group, ldx) <= pdap_smem_limit()) {
            s.group = group;
            s.variant = dp4;
            s.smem = pdap_smem_bytes(n, group, ldx);
            s.keys_gemm = dp4 == 0;
            return s;
        }
        group = 0;
    }
    // a few directions on a long array: one per SM, all of a CTA's threads on it in every step, keys resident
    // (n = 10,000, d = 5, 100 directions: 645 us per call against 672 with k_select_x, 682 with k_select;
    // n = 2,000: 600 against 584, so short arrays stay with k_select_x)
    if (group == 0 && dp4 && n > 4000 && rows > 0 && rows <= 2 * 152 && pdap_smem_bytes(n, 1, ldx) <= pdap_smem_limit()) {
        s.group = 1;
        s.variant = dp4;
        s.smem = pdap_smem_bytes(n, 1, ldx);
        s.keys_gemm = false;
        return s;
    }
    if (pdap_x_eligible(d) && group != PDAP_STREAM_CHOICE) {
        // keys re-formed from X: as many directions per CTA as its warps and shared memory take; fewer where the
        // request's rows would leave SMs without a CTA
        int G = SX_G;
        while (G > 1 && sel_smem(nb, G, d) > SX_SMEM) --G;
        const int64_t per_sm = (rows + 151) / 152;
        if (rows > 0 && per_sm < G) G = per_sm <= 2 ? 1 : (per_sm <= 4 ? std::min(G, 4) : G);
        s.group = G;
        s.variant = PDAP_WARP | d | (lg << 16);
        s.smem = sel_smem(nb, G, d);
        s.keys_gemm = false;
        return s;
    }
    // a task's keys are the least the keys scratch holds: fewer directions per task where those are many bytes
    s.group = n > 8000000 || (rows > 0 && rows < PDAP_KEYS_GROUP) ? 2 : PDAP_KEYS_GROUP;
    s.variant = PDAP_KEYS | (lg << 16);
    s.smem = sel_smem(nb, 1, 0);
    s.keys_gemm = true;
    return s;
}

}  // namespace rrs
