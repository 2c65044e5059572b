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
// A list that would not fit (many keys alike: repeated points, a dense core; or n beyond what the buckets resolve), a
// run at the edge of the range, or bounds that do not hold once the median is known send the direction to further
// passes (SelRef), which all such directions of a block share.
//
// nb is a power of two chosen by n (sel_buckets): about 16 n / nb keys are listed for D_P (normal data), which must
// fit (nb - 256) / 2 pairs, and each costs its warp some ten instructions; a histogram of nb costs two scans.
__host__ __device__ constexpr int sel_cap0(int nb) { return nb / 16 > 128 ? nb / 16 : 128; }   // median run and pick scratch (pairs)
__host__ __device__ constexpr int sel_run_max(int nb) { return nb / 16 > 256 ? nb / 16 : 256; }   // longest median run listed
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
    float sc, of;
    float dup;                     // median run too long to list: a value that the range's sample holds twice (sel_twice)
};

// What the runs step finds (the same in every thread of the group).
struct SelRuns {
    int fb;           // the median run is not listed
    int c_lo0;        // keys below the median run
    int cnt0;         // keys in it, |r - rc| <= wm; 0: not known
    int cnt;          // keys listed: the median run's (all or none) and the second runs'
    int c2;           // rank of a key among all minus its rank in the list: D_AP second run, D_P deviations
    float wm;
    // D_P: y values that bound the keys left out: between the second runs (il, ih), outside them (ol, oh)
    float il, ih, ol, oh;
    bool second;      // the second runs are listed
};
// And what only long runs need (kept where sel_long says so, in shared memory: the passes want the registers).
struct SelLong {
    int lb;           // listed keys below the median run
    // D_P second runs too long to list: ||r - rc| - sdd| <= sw holds scnt keys and leaves out sin keys between them
    int swin, scnt, sin;
    float sdd, sw;
};
__device__ __forceinline__ bool sel_long(const SelRuns& R, int nb) { return R.fb || !R.second || R.cnt0 > sel_cap0(nb); }

// Further passes for one direction: its state, kept in shared memory between the passes.  Each pass takes the
// candidates (keys inside a window of raw bucket values, or every key, whose value, y or |y - m|, lies in [xlo, xhi])
// and either counts them into RB sub-buckets, lists those of one sub-bucket run, or lists the indices of tied ones; and
// it notes the smallest and largest value and the smallest index of what it takes.  A sub-bucket of more keys than the
// list holds becomes the next interval, between its smallest and largest value, until it is listed or all its
// keys are equal.  The median comes first, then the spread.  Where the range's sample held a value twice and that lies
// in the median run, a cheaper pass comes first, which counts the keys below it and equal to it (repeated points).
//
// Measured, D_P, 1,000 queries, 5 rounds of 50 directions, 10,001 points in 10 dims: 5.6 ms where all points differ, 8.2
// with 30% of them one point (231 with one warp selecting a direction's ranks by itself, 15.4 with every key in shared
// memory, k_pdap2 of two directions), 15.8 with 30% of them in a core 10^-4 as wide as the rest (190, 15.5); 2.5 million
// normal points in 5 dims, 2 rounds of 1,000 directions: 38 ms (2,290; 960 with stored keys and 256 threads a direction).
struct SelRef {
    int op;                    // the next pass: RF_DONE (none), RF_COUNT, RF_LIST, RF_TIES, RF_PIVOT
    int win, dev, ranged;      // candidates in the window; values |y - m|; [xlo, xhi] leaves some out
    float w, dd, m, xlo, xhi;
    float blo, bsc;            // sub-bucket of v: (v - blo) * bsc within [0, 1], in RB steps
    int b1, b2, list;          // RF_LIST: the sub-bucket run, and whether it is listed
    int vmin, vmax, imin;      // what the pass found (rf_ord); RF_PIVOT: candidates below and equal
    int fill;
    int spread;                // the spread is sought (else the median)
    int rest;                  // the stage's second rank is sought by itself
    int cnt, r1, r2, below;    // candidates, ranks among them (r2 < 0: none), keys below them
    int q1, q2;                // the stage's ranks among its first candidates
    int alleq;                 // every key is equal
    float m1, m2, v1;
    int im1, im2, i1, nle;     // nle: keys not above the median
    SelRuns R;
    SelLong X;
};
constexpr int RF_DONE = 0, RF_COUNT = 1, RF_LIST = 2, RF_TIES = 3, RF_PIVOT = 4, RB = 256, RF_PASSES = 160;

template <int NG>
struct CtlS {
    int red[NG][NWARP / NG];
    float fred[NG][2 * NWARP / NG];   // two per warp of a group
    int fill[NG][2];
    int f_b1[NG], f_c1[NG], f_b2[NG], f_c2[NG];
    float pv1[NG], pv2[NG];
    int pi1[NG], pi2[NG];
    int gn[NG], gi[NG];
    SelPar par[NG];
    SelRef rf[NG];
};

// two k_select_x CTAs, with the 1 KB that each reserves, fill the 228 KB of an SM at most
static_assert(2 * (SX_SMEM + sizeof(CtlS<SX_G>) + 1024) <= 228 * 1024, "k_select_x: two CTAs per SM");

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
// direction to further passes, which are the tail of its launch: with one group of 32 and 2 interquartile ranges that
// was 1 of 2,500 normal directions, with four groups it is below 1 in 10^6.
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

// A value that the range's sample holds twice, not a number if there is none; of several the one nearest below its middle.
template <class K>
__device__ __noinline__ float sel_twice(const K y, int n)
{
    const int lane = threadIdx.x & 31;
    float dup = __int_as_float(0x7FC00000);
#pragma unroll 1
    for (int k = 0; k < RS; ++k) {
        const float v = warp_sort(y.get(sel_sample(n, lane, k))), next = __shfl_down_sync(0xFFFFFFFFu, v, 1);
        const unsigned twice = __ballot_sync(0xFFFFFFFFu, v == next && lane < 31), low = twice & 0xFFFFu;
        if (twice) dup = __shfl_sync(0xFFFFFFFFu, v, low ? 31 - __clz(low) : __ffs(twice) - 1);
    }
    return dup;
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

// The key of a scaled value v: (v - (of - 2^23)) / sc, a few roundings off: moved by 16 ulp towards dir.
__device__ __forceinline__ float sel_edge(const SelPar& par, float v, float dir)
{
    const float o = par.of - TWO23, inv = __fdiv_rn(1.0f, par.sc), a = (v - o) * inv;
    return a + dir * 2e-6f * (fabsf(a) + fabsf(o * inv) + fabsf(v * inv));
}

// The smallest s with more than rk keys in the buckets [ba - s, bb + s], where that is below ss: walked down from there,
// 32 at a time, over a gap with no keys that is rarely longer.  By a warp.
__device__ __noinline__ int sel_below_gap(const unsigned* H, int nb, int ba, int bb, int ss, int rk)
{
    const int lane = threadIdx.x & 31;
    for (;;) {
        const int s = ss - 1 - lane;
        const bool more = s >= 0 && (int)H[min(bb + s, nb - 1)] - (ba - s >= 1 ? (int)H[ba - s - 1] : 0) > rk;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, more);
        if (m != 0xFFFFFFFFu) return ss - __popc(m);
        ss -= 32;
    }
}

// Runs of one direction from its prefix counts, and its gather windows.  Windows are symmetric about an integer
// bucket: a median run of an even number of buckets takes one more above.
//
// D_P: let ss be the smallest s with more than k2 keys in the buckets [ba - s, bb + s], s1 the smallest with more than
// k1, w = bb - ba + 1.  A bucket b holds the keys of scaled value within 1/2 of b and the median m lies in the median
// run, so the MAD ranks' deviations are not below s1 - 1 and not above ss + w bucket widths: the keys that hold those
// ranks lie within w + 1 buckets of what is between bb + s1 and bb + ss, or ba - ss and ba - s1.  (With ss alone, an even
// n whose two ranks lie in different buckets left the lower one out: 0.4% of the directions of 698 normal points, each
// two more passes.)  The keys left out between the runs and outside them are bounded by the runs' edges, which sel_picks
// compares with the deviations it picks.
__device__ __forceinline__ SelRuns sel_runs(const unsigned* H, int nb, int n, bool ap, SelPar& par, SelLong& X)
{
    const int lane = threadIdx.x & 31;
    const int k1 = (n - 1) / 2, k2 = n / 2, cap1 = (nb - NB2) / 2;
    auto P = [&](int b) { return b < 0 ? 0 : (int)H[b]; };
    SelRuns R{};
    X = SelLong{};
    const int ba = sel_find(H, nb, (unsigned)k1);
    int bb = k2 == k1 ? ba : sel_find(H, nb, (unsigned)k2);
    bb += (ba + bb) & 1;
    par.w0 = par.w1 = -1.0f;
    par.dd = 0.0f;
    par.nrc2 = 0ull;
    R.fb = 1;
    if (ba < 1 || bb > nb - 2) return R;   // an edge bucket holds every key beyond the range
    R.c_lo0 = P(ba - 1);
    R.cnt0 = P(bb) - R.c_lo0;
    R.fb = R.cnt0 > sel_run_max(nb);
    const int own = R.fb ? 0 : R.cnt0;   // of the median run listed
    R.cnt = own;
    const int mid = (ba + bb) / 2;
    par.nrc2 = dup2(-(TWO23 + (float)mid));
    R.wm = (float)(bb - mid);
    if (!R.fb) par.w0 = R.wm;
    if (ap) {
        // keys above the median if none ties it; where the run is too long to list, if all of the run ties it (the few
        // that do not move the ranks by half their number: one bucket more on either side)
        const int npos = R.fb ? n - (R.c_lo0 + R.cnt0) : ((n & 1) ? (n - 1) / 2 : n / 2);
        if (npos > 0) {
            const int gb = n - npos;
            int b3 = sel_find(H, nb, (unsigned)(gb + (npos - 1) / 2));
            int b4 = (npos & 1) ? b3 : sel_find(H, nb, (unsigned)(gb + npos / 2));
            if (R.fb) {
                b3 = max(b3 - 1, bb + 1);
                ++b4;
            }
            if (b3 <= bb) {   // the runs meet: one window around both
                const int hw = max(b4, bb) - mid, lo = mid - hw, hi = mid + hw;
                if (lo >= 1 && hi <= nb - 2) {
                    const int below = P(lo - 1);
                    R.second = P(hi) - below <= cap1;
                    if (R.second) {
                        R.cnt = P(hi) - below;
                        R.c2 = below;
                        X.lb = R.c_lo0 - below;
                        par.w0 = (float)hw;
                    }
                }
            } else {
                b4 += (b3 + b4) & 1;
                if (b4 <= nb - 2) {
                    const int c1 = P(b4) - P(b3 - 1);
                    R.second = c1 + own <= cap1;
                    if (R.second) {
                        R.cnt = c1 + own;
                        R.c2 = P(b3 - 1) - own;   // the listed keys below the run are the median run's
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
    int s1 = ss;
    if (k1 != k2 && ss > 0 && win(ss - 1) > k1) s1 = sel_below_gap(H, nb, ba, bb, ss, k1);
    const int hw = bb - ba + 2;
    const int L0 = ba - ss - hw, L1 = ba - s1 + hw, R0 = bb + s1 - hw, R1 = bb + ss + hw;
    if (L0 >= 1 && R1 <= nb - 2) {
        const bool apart = L1 < ba;
        const int pl = P(L0 - 1), all = P(R1) - pl, left_out = apart ? P(R0 - 1) - P(L1) : 0;
        const float sdd = apart ? 0.5f * (float)(R0 + R1) - (float)mid : 0.0f;
        const float sw = apart ? 0.5f * (float)(R1 - R0) : (float)(R1 - mid);
        // the list holds the second runs and the median run; where that is not listed and the runs meet it, nothing
        const int more = apart ? own : 0, nlist = all - left_out + more;
        if (nlist <= cap1 && !(R.fb && !apart)) {
            R.second = true;
            R.cnt = nlist;
            R.c2 = left_out - more;
            X.lb = P(apart ? L1 : ba - 1) - pl;
            if (apart) {
                par.dd = sdd;
                par.w1 = sw;
            } else {
                par.w0 = sw;
            }
        } else {
            X.swin = 1;
            X.sin = left_out;
            X.scnt = all - left_out;
            X.sdd = sdd;
            X.sw = sw;
        }
        R.il = sel_edge(par, (float)L1 + 0.5f, -1.0f);
        R.ih = sel_edge(par, (float)R0 - 0.5f, 1.0f);
        R.ol = sel_edge(par, (float)L0 - 0.5f, 1.0f);
        R.oh = sel_edge(par, (float)R1 + 0.5f, -1.0f);
    }
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

// Floats as ints of the same order, for integer atomics (-0 just below +0).
__device__ __forceinline__ int rf_ord(float v)
{
    const int b = __float_as_int(v);
    return b < 0 ? b ^ 0x7FFFFFFF : b;
}
__device__ __forceinline__ float rf_val(int o) { return __int_as_float(o < 0 ? o ^ 0x7FFFFFFF : o); }

constexpr int TIE_MAX = 768;   // larger groups of equal values are taken at their smallest index, as k_pdap2 does

// Ranks s1 <= s2 of the list (B, I) of cnt pairs, by value and then by point index (a group of more than TIE_MAX equal
// values: its smallest index), by bisection over the value and then the index: some 60 walks of the list, where ranking
// every pair against all others takes cnt of them (1,800 pairs of one warp: 3,500 steps against 100,000).
template <int GS, class CT>
__device__ __noinline__ void sel_bisect(const Grp<GS> q, const float* B, const int* I, int cnt, int s1, int s2, CT& C,
                                        float& v1, float& v2, int& i1, int& i2)
{
    auto count = [&](auto f) {
        int c = 0;
        for (int t = q.t; t < cnt; t += GS) c += f(t);
        if (GS == 32) return (int)__reduce_add_sync(0xFFFFFFFFu, c);
        return gsum(q, c, C);
    };
    auto ord = [&](int t) { return rf_ord(__fadd_rn(B[t], 0.0f)); };   // -0 counts as 0
    auto nth = [&](int s, float& v, int& iv) {
        int lo = INT_MIN, hi = INT_MAX;   // the smallest value not above which lie more than s
        while (lo < hi) {
            const int mid = (int)(((int64_t)lo + hi) >> 1);
            if (count([&](int t) { return ord(t) <= mid; }) > s) hi = mid;
            else lo = mid + 1;
        }
        const int o = lo, below = count([&](int t) { return ord(t) < o; }), same = count([&](int t) { return ord(t) == o; });
        const int r = same > TIE_MAX ? 0 : s - below;
        lo = 0;
        hi = INT_MAX;
        while (lo < hi) {
            const int mid = lo + (hi - lo) / 2;
            if (count([&](int t) { return ord(t) == o && I[t] <= mid; }) > r) hi = mid;
            else lo = mid + 1;
        }
        v = rf_val(o);
        iv = lo;
    };
    nth(s1, v1, i1);
    v2 = v1;
    i2 = i1;
    if (s2 != s1) nth(s2, v2, i2);
}
template <int GS, class CT>
__device__ __forceinline__ void sel_rank(const Grp<GS>& q, const float* B, const int* I, int cnt, int s1, int s2, CT& C,
                                         float& v1, float& v2, int& i1, int& i2)
{
    // a larger group ranks pairs side by side, and its walks end in barriers: n = 100,000, d = 100, runs of about 150
    // pairs and 128 threads, 60.2 against 61.4 ms
    if (cnt <= (GS == 32 ? 192 : 512)) gpick(q, B, I, cnt, s1, s2, C, v1, v2, i1, i2);
    else sel_bisect<GS, CT>(q, B, I, cnt, s1, s2, C, v1, v2, i1, i2);
}

// The spread's picks from a direction's list once its median (m1, m2) is known, nle keys not above it (D_AP), by a group;
// false where the list does not hold them for sure (its keys may have become deviations by then).
template <int GS, class CT>
__device__ __forceinline__ bool sel_spread(const Grp<GS>& q, const SelRuns& R, const SelPar& par, CT& C, unsigned* H, int nb,
                                           int n, bool ap, float m1, float m2, int nle, int& ip1, int& ip2)
{
    constexpr int TCAP = 128;
    if (!R.second) return false;
    const int cap0 = sel_cap0(nb), cap1 = (nb - NB2) / 2;
    float* TB = reinterpret_cast<float*>(H + nb);
    int* TI = reinterpret_cast<int*>(TB + cap0);
    float* B = reinterpret_cast<float*>(H + NB2);
    int* I = reinterpret_cast<int*>(H + NB2 + cap1);
    float p1, p2;
    if (ap) {
        const int npos = n - nle, s3 = nle + (npos - 1) / 2 - R.c2, s4 = nle + npos / 2 - R.c2;
        // the listed keys of the second run are the list's last ones in rank
        if (s3 < (par.w1 < 0.0f || R.fb ? 0 : R.cnt0) || s4 >= R.cnt) return false;   // not the positive count of the guess
        float lo = FLT_MAX, hi = -FLT_MAX;
        for (int t = q.t; t < R.cnt; t += GS) {
            lo = fminf(lo, B[t]);
            hi = fmaxf(hi, B[t]);
        }
        gminmax(q, lo, hi, C, lo, hi);
        if (!gpick_bins<GS, CT, TCAP>(q, B, I, R.cnt, s3, s4, lo, hi, H, TB, TI, C, p1, p2, ip1, ip2))
            sel_bisect<GS, CT>(q, B, I, R.cnt, s3, s4, C, p1, p2, ip1, ip2);
        return true;
    }
    const float m = __fmul_rn(__fadd_rn(m1, m2), 0.5f);
    for (int t = q.t; t < R.cnt; t += GS) B[t] = fabsf(__fsub_rn(B[t], m));
    q.sync();
    // deviations of the keys left out: at most inner between the runs, at least outer outside them
    const float inner = R.c2 ? fmaxf(__fsub_rn(m, R.il), __fsub_rn(R.ih, m)) : -1.0f;
    const float outer = fminf(__fsub_rn(m, R.ol), __fsub_rn(R.oh, m));
    const int s1 = (n - 1) / 2 - R.c2, s2 = n / 2 - R.c2;
    if (s1 < 0 || s2 >= R.cnt || !(inner < outer)) return false;
    // picks within [inner, outer], or other passes find them: a histogram over that range serves
    if (!gpick_bins<GS, CT, TCAP>(q, B, I, R.cnt, s1, s2, fmaxf(inner, 0.0f), outer, H, TB, TI, C, p1, p2, ip1, ip2))
        sel_bisect<GS, CT>(q, B, I, R.cnt, s1, s2, C, p1, p2, ip1, ip2);
    return inner < p1 && outer > p2;   // strictly: no key left out ties a pick
}

// Sets a direction's next pass, by its warp: sub-buckets between blo and bhi, one for everything where that is no
// interval.
__device__ __forceinline__ void rf_count(SelRef& F, unsigned* H, float blo, float bhi)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    for (int b = lane; b < RB; b += 32) H[b] = 0u;
    if (lane == 0) {
        float sc = __fdiv_rn(1.0f, __fsub_rn(bhi, blo));
        if (!(bhi > blo) || !(fabsf(blo) <= FLT_MAX) || !(sc > 0.0f)) sc = blo = 0.0f;
        F.op = RF_COUNT;
        F.blo = blo;
        F.bsc = sc <= FLT_MAX ? sc : FLT_MAX;
        F.vmin = INT_MAX;
        F.vmax = INT_MIN;
        F.imin = INT_MAX;
    }
    __syncwarp();
}

// Candidates of a stage: cnt of them, below keys under them, the stage's ranks q1 <= q2 among them.
__device__ __forceinline__ void rf_stage(SelRef& F, int win, float w, float dd, float xlo, int cnt, int below, int q1, int q2)
{
    if ((threadIdx.x & 31) == 0) {
        F.win = win;
        F.w = w;
        F.dd = dd;
        F.xlo = xlo;
        F.xhi = FLT_MAX;
        F.ranged = xlo > -FLT_MAX && !F.dev;   // deviations are never below the lowest xlo, 0
        F.cnt = cnt;
        F.below = below;
        F.q1 = F.r1 = q1;
        F.q2 = q2;
        F.r2 = q2 != q1 ? q2 : -1;
        F.rest = 0;
    }
}

// Start of the median's passes: the run that was too long to list, or every key.  pivot: a value met twice may be tried.
__device__ __forceinline__ void rf_median(SelRef& F, const SelPar& par, unsigned* H, int nb, int n, bool every, bool pivot)
{
    const SelRuns& R = F.R;
    const int k1 = (n - 1) / 2, k2 = n / 2;
    const bool win = R.cnt0 > 0 && !every;
    const float mid = -(lo_f(par.nrc2) + TWO23);
    const float lo = win ? sel_edge(par, mid - R.wm - 0.5f, -1.0f) : sel_edge(par, 0.0f, -1.0f);
    const float hi = win ? sel_edge(par, mid + R.wm + 0.5f, 1.0f) : sel_edge(par, (float)nb, 1.0f);
    if ((threadIdx.x & 31) == 0) F.spread = F.dev = 0;
    if (win) rf_stage(F, 1, R.wm, 0.0f, -FLT_MAX, R.cnt0, R.c_lo0, k1 - R.c_lo0, k2 - R.c_lo0);
    else rf_stage(F, 0, 0.0f, 0.0f, -FLT_MAX, n, 0, k1, k2);
    rf_count(F, H, lo, hi);
    const float at = __fadd_rn(__fmaf_rn(par.dup, par.sc, par.of), lo_f(par.nrc2));
    if (pivot && win && fabsf(at) <= R.wm && (threadIdx.x & 31) == 0) {
        F.op = RF_PIVOT;
        F.xlo = par.dup;
        F.vmin = F.vmax = 0;
    }
    __syncwarp();
}

// Start of the spread's passes once the median is known (F.m1, F.m2, F.nle): D_AP the keys above it, D_P the second
// runs that were too long to list, or every deviation.
__device__ __forceinline__ void rf_spread(SelRef& F, const SelPar& par, unsigned* H, int nb, int n, bool ap, bool every)
{
    const SelRuns& R = F.R;
    const float m1 = F.m1, m = __fmul_rn(__fadd_rn(m1, F.m2), 0.5f);
    const int k1 = (n - 1) / 2, k2 = n / 2, npos = n - F.nle;
    const float top = sel_edge(par, (float)nb, 1.0f);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        F.spread = 1;
        F.dev = !ap;
        F.m = m;
    }
    if (ap) {
        const int b = __float_as_int(m1);
        const float above = m1 >= 0.0f ? __int_as_float((b & 0x7FFFFFFF) + 1) : __int_as_float(b - 1);   // next value up
        rf_stage(F, 0, 0.0f, 0.0f, above, npos, F.nle, (npos - 1) / 2, npos / 2);
        rf_count(F, H, m1, top);
        return;
    }
    const SelLong& X = F.X;
    const bool swin = !every && !R.second && X.swin;
    const float inner = swin && X.sin ? fmaxf(__fsub_rn(m, R.il), __fsub_rn(R.ih, m)) : -1.0f;
    const float outer = fminf(__fsub_rn(m, R.ol), __fsub_rn(R.oh, m));
    if (swin && k1 >= X.sin && k2 - X.sin < X.scnt && inner < outer) {
        rf_stage(F, 1, X.sw, X.sdd, 0.0f, X.scnt, X.sin, k1 - X.sin, k2 - X.sin);
        rf_count(F, H, fmaxf(inner, 0.0f), outer);
    } else {
        rf_stage(F, 0, 0.0f, 0.0f, 0.0f, n, 0, k1, k2);
        rf_count(F, H, 0.0f, __fmul_rn(0.5f, __fsub_rn(top, sel_edge(par, 0.0f, -1.0f))));
    }
}

// Indices of up to TIE_MAX ties: first where the median run's list goes, then in the sub-buckets' memory; 16 bits each
// for clouds of up to 32,000 points (nb <= 2,048, sel_buckets), whose lists are the shorter ones.
__device__ __forceinline__ void rf_tie_put(unsigned* H, int nb, int t, unsigned i)
{
    const int cap = 2 * sel_cap0(nb);
    if (nb <= 2048) reinterpret_cast<uint16_t*>(t < 2 * cap ? H + nb : H - cap)[t] = (uint16_t)i;
    else (t < cap ? H + nb : H - cap)[t] = i;
}
__device__ __forceinline__ int rf_tie(const unsigned* H, int nb, int t)
{
    const int cap = 2 * sel_cap0(nb);
    if (nb <= 2048) return reinterpret_cast<const uint16_t*>(t < 2 * cap ? H + nb : H - cap)[t];
    return (int)(t < cap ? H + nb : H - cap)[t];
}

// The sub-bucket of rank r among the RB counters: its number b, the candidates below it c, those in it h; total: all.
__device__ __forceinline__ void rf_find(const unsigned* H, int r, int& b, int& c, int& h, int& total)
{
    constexpr int PER = RB / 32;
    const int lane = threadIdx.x & 31;
    int v[PER], own = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        v[k] = (int)H[lane * PER + k];
        own += v[k];
    }
    int incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    int at = 0, below = incl - own, in = v[0];
#pragma unroll
    for (int k = 1; k < PER; ++k)
        if (below + in <= r && at == k - 1) {
            below += in;
            in = v[k];
            at = k;
        }
    const unsigned has = __ballot_sync(0xFFFFFFFFu, incl > r);
    const int src = has ? __ffs(has) - 1 : 31;
    b = __shfl_sync(0xFFFFFFFFu, lane * PER + at, src);
    c = __shfl_sync(0xFFFFFFFFu, below, src);
    h = __shfl_sync(0xFFFFFFFFu, in, src);
}

// A direction's step after a pass, by one warp: the next pass, or its picks written and RF_DONE.
template <class CT>
__device__ __noinline__ void rf_step(CT& C, int g, unsigned* H, int nb, int n, bool ap, int pass, ResDev* out, int* err)
{
    const int lane = threadIdx.x & 31, cap0 = sel_cap0(nb);
    SelRef& F = C.rf[g];
    const SelPar& par = C.par[g];
    const Grp<32> q{g, lane};
    float* TB = reinterpret_cast<float*>(H + nb);
    int* TI = reinterpret_cast<int*>(TB + cap0);
    const int op = F.op, fill = F.fill, spread = F.spread, win = F.win, found1 = F.vmin, found2 = F.vmax;
    int r1 = F.r1, r2 = F.r2, cnt = F.cnt, below = F.below;
    const bool one = op == RF_PIVOT || op == RF_TIES;   // a pass for the one value xlo
    const float vmin = one ? F.xlo : rf_val(found1), vmax = one ? vmin : rf_val(found2);
    float v1 = vmin, v2 = vmin;   // the ranks' values and point indices, once found
    int i1 = -1, i2 = -1, le = 0;   // le: candidates not above v1
    bool found = false, tie = false, bad = pass >= RF_PASSES;
    __syncwarp();
    if (op == RF_PIVOT) {
        // ranks among the keys equal to the value tried, or the passes without it
        const int a1 = below + r1 - found1, a2 = below + r2 - found1;
        if (a1 < 0 || a1 >= found2) {
            rf_median(F, par, H, nb, n, false, false);
            return;
        }
        r1 = a1;
        if (r2 >= 0) r2 = a2 < found2 ? a2 : -1;
        cnt = found2;
        below = found1;
        tie = true;
        if (lane == 0) {
            F.r1 = r1;
            F.r2 = r2;
            F.cnt = cnt;
            F.below = below;
        }
    } else if (op == RF_COUNT) {
        int b, c, h, b2, c2, h2, total;
        rf_find(H, r1, b, c, h, total);
        b2 = b;
        c2 = c;
        h2 = h;
        if (r2 >= 0) rf_find(H, r2, b2, c2, h2, total);
        bad |= total != cnt;
        if (!bad) {
            if (vmin == vmax) {
                tie = true;
            } else {
                const int both = c2 + h2 - c;   // no candidate lies between the two ranks' sub-buckets
                const bool two = r2 >= 0 && (b2 == b || both <= cap0);
                const int in = two ? both : h;
                if (in == cnt && in > cap0) {   // all in one sub-bucket: narrow the range first
                    if (lane == 0) {
                        F.xlo = vmin;
                        F.xhi = vmax;
                        F.ranged = 1;
                    }
                    rf_count(F, H, vmin, vmax);
                    return;
                }
                if (lane == 0) {
                    F.op = RF_LIST;
                    F.b1 = b;
                    F.b2 = two ? b2 : b;
                    F.list = in <= cap0;
                    F.cnt = in;
                    F.below = below + c;
                    F.r1 = r1 - c;
                    F.r2 = two ? r2 - c : -1;
                    F.vmin = INT_MAX;
                    F.vmax = INT_MIN;
                    F.imin = INT_MAX;
                    F.fill = 0;
                }
                __syncwarp();
                return;
            }
        }
    } else if (op == RF_LIST) {
        if (F.list) {
            bad |= fill != cnt;
            if (!bad) {
                sel_rank<32, CT>(q, TB, TI, cnt, r1, r2 >= 0 ? r2 : r1, C, v1, v2, i1, i2);
                for (int t = lane; t < cnt; t += 32) le += TB[t] <= v1;
                le = __reduce_add_sync(0xFFFFFFFFu, le);
                found = true;
            }
        } else if (vmin == vmax) {
            tie = true;
        } else {
            if (lane == 0) {
                F.xlo = vmin;
                F.xhi = vmax;
                F.ranged = 1;
            }
            rf_count(F, H, vmin, vmax);
            return;
        }
    } else {
        // the indices of cnt ties: the ranks' ones by bisection over the index
        bad |= fill != cnt;
        if (!bad) {
            auto at = [&](int t) { return rf_tie(H, nb, t); };
            auto nth = [&](int r) {
                int lo = 0, hi = n - 1;
                while (lo < hi) {
                    const int mid = lo + (hi - lo) / 2;
                    int c = 0;
                    for (int t = lane; t < cnt; t += 32) c += at(t) <= mid;
                    if (__reduce_add_sync(0xFFFFFFFFu, c) > r) hi = mid;
                    else lo = mid + 1;
                }
                return lo;
            };
            i1 = i2 = nth(r1);
            if (r2 >= 0) i2 = nth(r2);
            le = cnt;
            found = true;
        }
    }
    if (tie && !bad) {
        // all candidates equal: by rank of their index, or the smallest one (groups of more than TIE_MAX, and of more
        // than 256 when every key is equal: k_pdap2's rules)
        const bool alleq = (!spread && cnt == n) || F.alleq;
        __syncwarp();
        if (lane == 0) F.alleq = alleq;
        le = cnt;
        if (cnt == 1 || cnt > (alleq ? 256 : TIE_MAX)) {
            i1 = i2 = F.imin;
            found = true;
        } else {
            if (lane == 0) {
                F.op = RF_TIES;
                F.xlo = F.xhi = vmin;
                F.ranged = 1;
                F.fill = 0;
            }
            __syncwarp();
            return;
        }
    }
    if (bad || !found) {
        // the counts do not add up (never seen), or no end: every key once more, then give up
        if (win && pass < RF_PASSES) {
            if (spread) rf_spread(F, par, H, nb, n, ap, true);
            else rf_median(F, par, H, nb, n, true, false);
            return;
        }
        if (lane == 0) {
            atomicOr(err, ERR_SELECT_ITER);
            put_picks(out, spread ? F.im1 : -1, spread ? F.im2 : -1, -1, -1);
            F.op = RF_DONE;
        }
        __syncwarp();
        return;
    }
    // one or both ranks found
    const bool rest = F.rest, split = F.q2 != F.q1 && r2 < 0 && !rest;
    const float w1 = rest ? F.v1 : v1, w2 = v2;
    const int j1 = rest ? F.i1 : i1, j2 = i2;
    if (split) {
        // the second rank lies in another sub-bucket: it is sought by itself, from the stage's first candidates
        const int nle = below + le;
        __syncwarp();
        if (!spread) rf_median(F, par, H, nb, n, !win, false);
        else rf_spread(F, par, H, nb, n, ap, !win);
        if (lane == 0) {
            F.v1 = v1;
            F.i1 = i1;
            if (!spread) F.nle = nle;
            F.r1 = F.q2;
            F.r2 = -1;
            F.rest = 1;
        }
        __syncwarp();
        return;
    }
    int nle = rest ? F.nle : below + le;
    if (spread) {
        bool ok = true;
        if (!ap && win) {
            const SelRuns& R = F.R;
            const float inner = F.X.sin ? fmaxf(__fsub_rn(F.m, R.il), __fsub_rn(R.ih, F.m)) : -1.0f;
            const float outer = fminf(__fsub_rn(F.m, R.ol), __fsub_rn(R.oh, F.m));
            ok = inner < w1 && outer > w2;
        }
        if (!ok) {
            __syncwarp();
            rf_spread(F, par, H, nb, n, ap, true);
            return;
        }
        if (lane == 0) put_picks(out, F.im1, F.im2, j1, j2);
    } else {
        __syncwarp();
        if (lane == 0) {
            F.m1 = w1;
            F.m2 = w2;
            F.im1 = j1;
            F.im2 = j2;
            F.nle = nle;
        }
        __syncwarp();
        int ip1 = NOPOS, ip2 = NOPOS;
        const bool none = ap && nle == n;
        const bool listed = C.fill[g][0] == F.R.cnt;   // else the list is not what the counts promise
        if (!none && !(listed && sel_spread(q, F.R, par, C, H, nb, n, ap, w1, w2, nle, ip1, ip2))) {
            __syncwarp();
            rf_spread(F, par, H, nb, n, ap, false);
            return;
        }
        if (lane == 0) put_picks(out, j1, j2, ip1, ip2);
    }
    if (lane == 0) F.op = RF_DONE;
    __syncwarp();
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

// The raw sub-bucket of a value (its number plus MAGIC), monotone: the edge ones take every value beyond them.
__device__ __forceinline__ int rf_raw(float v, float blo, float bsc)
{
    return __float_as_int(__fmaf_rn(__saturatef(__fmul_rn(__fsub_rn(v, blo), bsc)), (float)(RB - 1), TWO23));
}
__device__ __forceinline__ void rf_red(unsigned hb, int raw, bool take)
{
    asm volatile("{\n .reg .pred p;\n setp.ne.s32 p, %1, 0;\n @p red.shared.add.u32 [%0], 1;\n}" ::"r"(hb + 4u * (unsigned)raw),
                 "r"((int)take));
}

// One direction's keys k of the points i, i + 1 (then i + 2, i + 3; the next four 128 further on) in the current pass, by
// a whole warp.  Bound by its instructions: a pass takes about as long as the first two together (10,000 points in 10
// dims, 50,000 directions: 1.0 ms against 1.1), RF_PIVOT less than half.  Where many keys are alike most candidates
// share a sub-bucket: those in the one of the warp's first count with one reduction.
template <int S>
__device__ __forceinline__ void rf_keys(SelRef& F, const SelPar& par, unsigned* H, int nb, const unsigned long long (&k)[S],
                                        unsigned i, unsigned n)
{
    const int lane = threadIdx.x & 31, op = F.op;
    const float nan = __int_as_float(0x7FC00000);
    auto at = [&](int j) { return i + 128 * (j >> 2) + (j & 3); };
    float v[2 * S];   // the candidates' values, others not a number
#pragma unroll
    for (int h = 0; h < S; ++h) {
        v[2 * h] = lo_f(k[h]);
        v[2 * h + 1] = hi_f(k[h]);
    }
    if (at(2 * S - 1) >= n) {   // the last points
#pragma unroll
        for (int j = 0; j < 2 * S; ++j)
            if (at(j) >= n) v[j] = nan;
    }
    if (op == RF_PIVOT) {
        const float x = F.xlo;
        unsigned lt = 0, eq = 0;
#pragma unroll
        for (int j = 0; j < 2 * S; ++j) {
            lt += v[j] < x;
            eq += v[j] == x;
        }
        if (eq && (int)i < F.imin) {
            int im = INT_MAX;
#pragma unroll
            for (int j = 2 * S - 1; j >= 0; --j)
                if (v[j] == x) im = (int)at(j);
            atomicMin(&F.imin, im);
        }
        const unsigned both = __reduce_add_sync(0xFFFFFFFFu, lt | eq << 16);
        if (lane == 0) {
            if (both & 0xFFFFu) atomicAdd(&F.vmin, (int)(both & 0xFFFFu));
            if (both >> 16) atomicAdd(&F.vmax, (int)(both >> 16));
        }
        return;
    }
    if (F.win) {
        const unsigned long long sc2 = par.sc2, of2 = par.of2, nrc2 = par.nrc2;
        const float w = F.w, dd = F.dd;
#pragma unroll
        for (int h = 0; h < S; ++h) {
            const unsigned long long t = add2(fma2(k[h], sc2, of2), nrc2);   // as sel_test rounds it
            if (!(fabsf(fabsf(lo_f(t)) - dd) <= w)) v[2 * h] = nan;
            if (!(fabsf(fabsf(hi_f(t)) - dd) <= w)) v[2 * h + 1] = nan;
        }
    }
    if (F.dev) {
        const float m = F.m;
#pragma unroll
        for (int j = 0; j < 2 * S; ++j) v[j] = fabsf(__fsub_rn(v[j], m));
    }
    if (F.ranged) {
        const float xlo = F.xlo, xhi = F.xhi;
#pragma unroll
        for (int j = 0; j < 2 * S; ++j)
            if (!(v[j] >= xlo && v[j] <= xhi)) v[j] = nan;
    }
    float lo = INFINITY, hi = -INFINITY;
#pragma unroll
    for (int j = 0; j < 2 * S; ++j) lo = fminf(lo, v[j]);
    const unsigned any = __ballot_sync(0xFFFFFFFFu, lo < INFINITY);
    if (!any) return;
    if (op == RF_TIES) {
#pragma unroll
        for (int j = 0; j < 2 * S; ++j)
            if (v[j] == v[j]) {
                const int pos = atomicAdd(&F.fill, 1);
                if (pos < TIE_MAX) rf_tie_put(H, nb, pos, at(j));
            }
        return;
    }
    const float blo = F.blo, bsc = F.bsc;
    if (op == RF_COUNT) {
        const int hot = __shfl_sync(0xFFFFFFFFu, rf_raw(lo, blo, bsc), __ffs(any) - 1);
        const unsigned hb = sel_base(H);
        unsigned c = 0;
#pragma unroll
        for (int j = 0; j < 2 * S; ++j) {
            const int raw = rf_raw(v[j], blo, bsc);
            const bool is = v[j] == v[j];
            c += is && raw == hot;
            rf_red(hb, raw, is && raw != hot);
        }
        c = __reduce_add_sync(0xFFFFFFFFu, c);
        if (lane == 0 && c) atomicAdd(&H[hot - MAGIC], c);
    } else {
        const int b1 = MAGIC + F.b1;
        const unsigned run = (unsigned)(F.b2 - F.b1);
        bool mine = false;
#pragma unroll
        for (int j = 0; j < 2 * S; ++j) {
            if (!(v[j] == v[j] && (unsigned)(rf_raw(v[j], blo, bsc) - b1) <= run)) v[j] = nan;
            mine |= v[j] == v[j];
        }
        if (!mine) return;
        if (F.list) {
            const int cap0 = sel_cap0(nb);
#pragma unroll
            for (int j = 0; j < 2 * S; ++j)
                if (v[j] == v[j])
                    sel_put(&F.fill, reinterpret_cast<float*>(H + nb), reinterpret_cast<int*>(H + nb) + cap0, cap0, v[j],
                            (int)at(j));
            return;
        }
        lo = INFINITY;
#pragma unroll
        for (int j = 0; j < 2 * S; ++j) lo = fminf(lo, v[j]);
    }
    if (lo < INFINITY) {
#pragma unroll
        for (int j = 0; j < 2 * S; ++j) hi = fmaxf(hi, v[j]);
        if (rf_ord(lo) < F.vmin) atomicMin(&F.vmin, rf_ord(lo));
        if (rf_ord(hi) > F.vmax) atomicMax(&F.vmax, rf_ord(hi));
        if ((int)i < F.imin) {   // rarely, once a candidate was met
            int im = INT_MAX;
#pragma unroll
            for (int j = 2 * S - 1; j >= 0; --j)
                if (v[j] == v[j]) im = (int)at(j);
            atomicMin(&F.imin, im);
        }
    }
}

// The picks of one direction from its list, by a group; false where further passes must find them: F then holds their
// start.  H: the direction's sel_words(nb) words, the list after NB2 words.
template <int GS, class CT>
__device__ __noinline__ bool sel_picks(const Grp<GS> q, const SelRuns R, const SelPar par, CT& C, unsigned* H, int nb,
                                       int n, bool ap, ResDev* out)
{
    const int k1 = (n - 1) / 2, k2 = n / 2, cap0 = sel_cap0(nb), cap1 = (nb - NB2) / 2;
    SelRef& F = C.rf[q.g];
    float* TB = reinterpret_cast<float*>(H + nb);
    int* TI = reinterpret_cast<int*>(TB + cap0);
    const float* B = reinterpret_cast<const float*>(H + NB2);
    const int* I = reinterpret_cast<const int*>(H + NB2 + cap1);
    auto start = [&] {   // of further passes, by the group's first thread
        F.R = R;
        F.alleq = 0;
        C.par[q.g] = par;
    };
    // the list must hold the keys the counts promise
    const bool listed = C.fill[q.g][0] == R.cnt;
    if (R.fb || !listed) {
        if (q.t == 0) start();
        q.sync();
        if (q.t < 32) rf_median(F, par, H, nb, n, !listed && !R.fb, true);
        return false;
    }
    float m1, m2;
    int im1, im2, ip1 = NOPOS, ip2 = NOPOS, nle = 0;
    if (R.cnt0 <= cap0) {
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
        sel_rank<GS, CT>(q, TB, TI, R.cnt0, k1 - R.c_lo0, k2 - R.c_lo0, C, m1, m2, im1, im2);
    } else {
        sel_bisect<GS, CT>(q, B, I, R.cnt, k1 - R.c_lo0 + F.X.lb, k2 - R.c_lo0 + F.X.lb, C, m1, m2, im1, im2);
    }
    if (ap) {
        // #(y <= med) = #(y <= m1): keys below the run plus its keys <= m1
        const bool apart = R.cnt0 <= cap0;
        int c = 0;
        for (int t = q.t; t < (apart ? R.cnt0 : R.cnt); t += GS) c += ((apart ? TB : B)[t] <= m1);
        nle = R.c_lo0 + gsum(q, c, C) - (apart ? 0 : F.X.lb);
    }
    if (!(ap && nle == n) && !sel_spread(q, R, par, C, H, nb, n, ap, m1, m2, nle, ip1, ip2)) {
        q.sync();
        if (q.t == 0) {
            start();
            F.m1 = m1;
            F.m2 = m2;
            F.im1 = im1;
            F.im2 = im2;
            F.nle = nle;
        }
        q.sync();
        if (q.t < 32) rf_spread(F, par, H, nb, n, ap, false);
        return false;
    }
    if (q.t == 0) put_picks(out, im1, im2, ip1, ip2);
    return true;
}

// The further passes of a block's directions, until none needs another; mine: this warp steps direction w.
template <class CT, class P>
__device__ __forceinline__ void sel_refine(const P& pass, CT& C, bool mine, int w, unsigned* H, int nb, int n, bool ap,
                                           ResDev* out, int* err)
{
    for (int it = 1;; ++it) {
        const bool busy = mine && C.rf[w].op != RF_DONE;
        if (!__syncthreads_or(busy)) return;
        pass();
        __syncthreads();
        if (busy) rf_step(C, w, H, nb, n, ap, it, out, err);
    }
}

// The further passes' functions take the kernels' parameters, not what those hold in registers by then.
template <int GS>
__device__ __noinline__ void sel_refine_k(const TaskDev* tasks, int G, const SlotDev* slots, const DsDev* dsets,
                                          ResDev* res, int* err, const float* kin, int nb, CtlS<1>& C)
{
    extern __shared__ __align__(16) unsigned sel_sm[];
    const int ti = blockIdx.x / G, g = blockIdx.x - ti * G;
    const TaskDev T = tasks[ti];
    const SlotDev& S = slots[T.slot];
    const int n = (int)dsets[T.ds].n;
    const float* y = kin + (size_t)blockIdx.x * ((n + 3) & ~3);
    unsigned* H = sel_sm;
    auto pass = [&] {
        // the row is padded to whole fours
        const unsigned t4 = 4 * threadIdx.x, w4 = t4 & ~127u;
        for (unsigned base = 0; base + w4 < (unsigned)n; base += 4 * GS) {   // whole warps
            const unsigned i = base + t4;
            ulonglong2 v = make_ulonglong2(0ull, 0ull);
            if (i < (unsigned)n) v = *reinterpret_cast<const ulonglong2*>(y + i);
            const unsigned long long k[2] = {v.x, v.y};
            rf_keys<2>(C.rf[0], C.par[0], H, nb, k, i, (unsigned)n);
        }
    };
    sel_refine(pass, C, threadIdx.x < 32, 0, H, nb, n, S.kind == 2, res + S.roff + T.j0 + g, err);
}

// Keys in device memory (kin: G x npad per task in launch order, formed by launch_pdap_keys): one block of GS
// threads per direction, so directions never wait for one another and a block's few barriers are its own.
// Measured at n = 10,000 (26,840 directions, 449 us): 30 instructions a key, the shared-memory pipe at 66% of its
// wavefronts (half of them the reductions), issue slots at 48%; warps wait for keys from memory first.
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
    SelLong X;
    const SelRuns R = sel_runs(H, nb, n, ap, par, X);
    if (sel_long(R, nb)) {
        if (q.t == 0) C.rf[0].X = X;
        if (R.fb && R.cnt0 > 0) par.dup = sel_twice(y, n);
    }
    q.sync();   // the histogram's memory takes the list from here
    if (par.w0 >= 0.0f || par.w1 >= 0.0f) {
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
    if (!R.fb && (ap || R.second) && R.cnt <= 32 * FJ && R.cnt0 <= 32 && C.fill[0][0] == R.cnt) {   // the same in every thread
        if (q.t < 32) {
            const bool ok = sel_picks_warp(R, par, H, nb, n, ap, out);
            if (q.t == 0) C.gi[0] = ok;
        }
        q.sync();
        if (C.gi[0]) return;
        q.sync();
    }
    if (!sel_picks<GS, CtlS<1>>(q, R, par, C, H, nb, n, ap, out))
        sel_refine_k<GS>(tasks, G, slots, dsets, res, err, kin, nb, C);
}

// A key is two half chains over the dims, added (key_halves), here without the zero-padded terms (a zero product
// leaves a chain unchanged): the values the other selection kernels form.
template <int D>
struct HalfChains {
    static constexpr int DP4 = (D + 3) & ~3, H2 = DP4 / 2, E0 = D < H2 ? D : H2;
};

// One direction's keys re-formed one by one, for the range sample (any d <= 16; u: the
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
__device__ __forceinline__ void load_points(const float* Xt, const float* X32, int ldx, unsigned i, int n,
                                            unsigned long long (&xv)[D][S], int at)
{
    if (Xt) {
        const size_t colst = (size_t)((n + 31) & ~31);
#pragma unroll
        for (int l = 0; l < D; ++l) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(Xt + l * colst + i);
            xv[l][at] = v.x;
            xv[l][at + 1] = v.y;
        }
        return;
    }
    constexpr int D4 = (D + 3) & ~3;
    float x[4][D4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4* xr = reinterpret_cast<const float4*>(X32 + (int64_t)min(i + k, (unsigned)n - 1u) * ldx);
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

// Further passes of k_select_x, for the directions that need them together: the keys of each formed as in its passes.
template <int D>
__device__ __noinline__ void sel_refine_x(const TaskDev* tasks, const SlotDev* slots, const DsDev* dsets, ResDev* res,
                                          int* err, int nb, int G, CtlS<SX_G>& C)
{
    using PG = PointGroups<D>;
    constexpr int DU = (D + 1) & ~1, NG = PG::NG, S2 = 2 * NG;
    extern __shared__ __align__(16) unsigned sel_sm[];
    const TaskDev T = tasks[blockIdx.x];
    const SlotDev& S = slots[T.slot];
    const float *Xt = dsets[T.ds].Xt, *X32 = dsets[T.ds].X32;
    const int n = (int)dsets[T.ds].n, ldx = dsets[T.ds].ldx, GA = T.nj;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, words = sel_words(nb), nwarps = blockDim.x >> 5;
    unsigned* area = sel_sm;
    const float2* uS = reinterpret_cast<const float2*>(area + (size_t)G * words);
    auto pass = [&] {
        for (unsigned base = w * PG::CHUNK; base < (unsigned)n; base += nwarps * PG::CHUNK) {
            const unsigned i = base + 4 * lane;
            unsigned long long xv[D][S2] = {};
#pragma unroll
            for (int p = 0; p < NG; ++p)
                if (i + 128 * p < (unsigned)n) load_points<D, S2>(Xt, X32, ldx, i + 128 * p, n, xv, 2 * p);
#pragma unroll 1
            for (int g = 0; g < GA; ++g) {
                if (C.rf[g].op == RF_DONE) continue;
                unsigned long long k[S2];
                form_keys<D, S2>(uS + g * DU, xv, k);
                rf_keys<S2>(C.rf[g], C.par[g], area + g * words, nb, k, i, (unsigned)n);
            }
        }
    };
    sel_refine(pass, C, w < GA, w, area + w * words, nb, n, S.kind == 2, res + S.roff + T.j0 + w, err);
}

// d <= 16: keys re-formed from X at both passes.  The whole CTA walks the points, four per thread with their
// coordinates in registers, and forms their keys for every direction of the task (packed FMAs over point pairs,
// the direction's pairs from shared memory); warp g then takes direction g's steps between the passes alone.
// X is read twice per task whatever its number of directions, and no key is stored, so 16 directions are in flight
// per SM at any n.  Measured at n = 10,000, d = 10 (10,000 directions, 247 us): 43 instructions a key over both passes,
// the shared-memory pipe at 53% of its wavefronts (two fifths of them the reductions), issue slots at 50% with the 16
// warps an SM holds.
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
            C.rf[w].op = RF_DONE;
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
            if (i + 128 * p < (unsigned)n) load_points<D, S2>(Dd.Xt, Dd.X32, ldx, i + 128 * p, n, xv, 2 * p);
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

    // the runs' record: held in registers through the next pass where the coordinates leave room for it, else in shared
    // memory (n = 10,000, d = 10: 22.4 against 24.9 ms with spills; a short pass feels the way there and back: n = 599,
    // d = 4 10.5 against 10.7 ms)
    constexpr bool HELD = D <= 6;
    SelRuns held{};
    unsigned* H = area + w * words;
    if (w < GA) {
        sel_prefix(q, H, nb, C);
        SelLong X;
        const SelRuns R = sel_runs(H, nb, n, ap, par, X);
        if (R.fb && R.cnt0 > 0) par.dup = sel_twice(y, n);
        if (HELD) held = R;
        if (lane == 0) {
            C.par[w] = par;
            if (!HELD) C.rf[w].R = R;
            if (sel_long(R, nb)) C.rf[w].X = X;
        }
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
                if (i + 128 * p < (unsigned)n) load_points<D, S2>(Dd.Xt, Dd.X32, ldx, i + 128 * p, n, xv, 2 * p);
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
    ResDev* out = res + S.roff + T.j0 + w;
    bool more = false;
    if (w < GA) {
        const SelRuns R = HELD ? held : C.rf[w].R;
        if (!HELD) par = C.par[w];
        const bool fast = !R.fb && (ap || R.second) && R.cnt <= 32 * FJ && R.cnt0 <= 32 && C.fill[w][0] == R.cnt &&
                          sel_picks_warp(R, par, H, nb, n, ap, out);
        more = !fast && !sel_picks<32, CtlS<SX_G>>(q, R, par, C, H, nb, n, ap, out);
    }
    if (__syncthreads_or(more)) sel_refine_x<D>(tasks, slots, dsets, res, err, nb, G, C);
}

// Buckets per direction by n: about 16 n / nb keys are listed for D_P and 0.001 x 2048 / nb x n lie in a bucket
// at the median (normal data), so up to about 1.9 million points these lines keep both well inside their buffers while
// the histograms stay small enough for 16 (k_select_x: nb = 2,048, 147 KB) or some 20 (k_select) directions per SM.
// Beyond that every direction takes further passes (SelRef), five in all where two would do.
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
