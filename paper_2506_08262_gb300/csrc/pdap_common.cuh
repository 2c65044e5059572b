// Device helpers shared by the selection kernels (pdap.cu, pdap_select.cu): thread groups, bucket maps, ranking of
// gathered pairs, and the iterated bucket selection every kernel falls back to.
#pragma once
#include <cuda_runtime.h>
#include <float.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include "rrs_internal.h"

namespace rrs {
namespace {

constexpr int NWARP = 32;    // largest warp count of a CTA
constexpr int NB = 2048;     // buckets per direction of k_pdap2
constexpr int CAP = 256;     // gathered keys per direction: the median run (and the D_AP MAD_+ run)
constexpr int CAP1 = 512;    // second gather buffer: the D_AP MAD_+ run or the D_P MAD runs L, R
constexpr int CAP1H = (NB - 256) / 2;   // D_P runs too large for it: pairs in the histogram area (after 256 counters)
constexpr int FB_NB = NB;    // fallback histogram (reuses the bucket area)
constexpr int FB_CAP = CAP + CAP1;  // fallback gather buffer: a direction's two gather areas

struct TrueT {
    static constexpr bool value = true;
};
struct FalseT {
    static constexpr bool value = false;
};

// A thread group working on one direction.  Groups of one warp need no barrier.  Larger ones are the parts of a block
// (k_pdap2: named barrier 1 + g) or, in a translation unit that defines PDAP_BLOCK_GROUPS, whole blocks: a barrier
// whose number is not a constant makes a block reserve all 16, and four such blocks fill an SM.
template <int GS>
struct Grp {
    int g, t;   // direction (group) index, thread index within the group
    __device__ __forceinline__ void sync() const
    {
        if constexpr (GS == 32)
            __syncwarp();
        else
#ifdef PDAP_BLOCK_GROUPS
            __syncthreads();
#else
            asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(GS) : "memory");
#endif
    }
};

template <int NBK = NB>
__device__ __forceinline__ int bucket(float y, float lo, float scale)
{
    // (y - lo) * scale, rounded once, truncated: monotone in y
    const int b = __float2int_rz(__fmul_rn(__fsub_rn(y, lo), scale));
    return b < 0 ? 0 : (b > NBK - 1 ? NBK - 1 : b);
}

// Bucket maps of k_pdap2: y*sc + off rounded once to an integer by the FMA itself.  o23 is off + 2^23,
// so a result r in [2^23, 2^24) is an integer and its float bits are MAGIC + (r - 2^23).  bucket_raw
// returns those bits as an int: non-decreasing in y for every result that is not a negative float, and
// every negative float is a negative int.  bucket_m clamps them to [0, NBK): no float-to-integer
// conversion, monotone non-decreasing in y.  A run of buckets [b1, b2] is the set of raw values in
// [raw_lo(b1), raw_hi(b2)] (signed comparisons), the edge buckets taking every value clamped into them.
constexpr int MAGIC = 0x4B000000;   // float bits of 2^23
constexpr float TWO23 = 8388608.0f;
__device__ __forceinline__ int bucket_raw(float y, float sc, float o23) { return __float_as_int(__fmaf_rn(y, sc, o23)); }
template <int NBK = NB>
__device__ __forceinline__ int bucket_m(float y, float sc, float o23)
{
    return min(max(bucket_raw(y, sc, o23), MAGIC), MAGIC + NBK - 1) - MAGIC;
}
template <int NBK = NB>
__device__ __forceinline__ int raw_lo(int b)
{
    return b <= 0 ? INT_MIN : MAGIC + b;
}
template <int NBK = NB>
__device__ __forceinline__ int raw_hi(int b)
{
    return b >= NBK - 1 ? INT_MAX : MAGIC + b;
}

__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}
__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v = fminf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

// Group sum of one int per thread (every thread gets the total).
template <int GS, class CT>
__device__ __forceinline__ int gsum(const Grp<GS>& q, int c, CT& C)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
    if ((q.t & 31) == 0) C.red[q.g][q.t >> 5] = c;
    q.sync();
    int s = 0;
#pragma unroll
    for (int i = 0; i < GS / 32; ++i) s += C.red[q.g][i];
    q.sync();
    return s;
}

// Group min and max.
template <int GS, class CT>
__device__ void gminmax(const Grp<GS>& q, float lo, float hi, CT& C, float& olo, float& ohi)
{
    lo = warp_min(lo);
    hi = warp_max(hi);
    constexpr int NW = GS / 32;
    if ((q.t & 31) == 0) {
        C.fred[q.g][q.t >> 5] = lo;
        C.fred[q.g][NW + (q.t >> 5)] = hi;
    }
    q.sync();
    olo = C.fred[q.g][0];
    ohi = C.fred[q.g][NW];
#pragma unroll
    for (int i = 1; i < NW; ++i) {
        olo = fminf(olo, C.fred[q.g][i]);
        ohi = fmaxf(ohi, C.fred[q.g][NW + i]);
    }
    q.sync();
}

// Group min and max of two pairs at once (one barrier round for both).
template <int GS, class CT>
__device__ __forceinline__ void gminmax2(const Grp<GS>& q, float& lo1, float& hi1, float& lo2, float& hi2, CT& C)
{
    constexpr int NW = GS / 32;   // at most 16: 4 NW values fit the 2 NWARP cells of fred
    static_assert(4 * NW <= 2 * NWARP, "gminmax2 scratch");
    lo1 = warp_min(lo1);
    hi1 = warp_max(hi1);
    lo2 = warp_min(lo2);
    hi2 = warp_max(hi2);
    const int w = q.t >> 5;
    if ((q.t & 31) == 0) {
        C.fred[q.g][w] = lo1;
        C.fred[q.g][NW + w] = hi1;
        C.fred[q.g][2 * NW + w] = lo2;
        C.fred[q.g][3 * NW + w] = hi2;
    }
    q.sync();
    lo1 = C.fred[q.g][0];
    hi1 = C.fred[q.g][NW];
    lo2 = C.fred[q.g][2 * NW];
    hi2 = C.fred[q.g][3 * NW];
#pragma unroll
    for (int i = 1; i < NW; ++i) {
        lo1 = fminf(lo1, C.fred[q.g][i]);
        hi1 = fmaxf(hi1, C.fred[q.g][NW + i]);
        lo2 = fminf(lo2, C.fred[q.g][2 * NW + i]);
        hi2 = fmaxf(hi2, C.fred[q.g][3 * NW + i]);
    }
    q.sync();
}

// Exclusive scan of h[0..NB) by the group; the bucket holding rank ra and the
// one holding rank rb (ra <= rb, both below the total), with the keys below each.
template <int GS, class CT, int NBK = NB>
__device__ void gfind(const Grp<GS>& q, const unsigned* h, int ra, int rb, CT& C, int& ba, int& ca, int& bb, int& cb)
{
    constexpr int PER = NBK / GS;   // 4 .. 32 consecutive buckets per thread, read as uint4
    static_assert(PER >= 4 && PER % 4 == 0, "gfind reads whole uint4");
    const int lane = q.t & 31, w = q.t >> 5;
    int own = 0;
    unsigned v[PER];
    const uint4* h4 = reinterpret_cast<const uint4*>(h + q.t * PER);
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
        if (hk > 0) {
            if (c <= ra && ra < c + hk) {
                C.f_b1[q.g] = q.t * PER + k;
                C.f_c1[q.g] = c;
            }
            if (c <= rb && rb < c + hk) {
                C.f_b2[q.g] = q.t * PER + k;
                C.f_c2[q.g] = c;
            }
        }
        c += hk;
    }
    q.sync();
    ba = C.f_b1[q.g];
    ca = C.f_c1[q.g];
    bb = C.f_b2[q.g];
    cb = C.f_c2[q.g];
    q.sync();
}

// Values and point indices of the 0-based ranks s1 <= s2 among the pairs (buf, ib)[0..cnt), ordered by
// value and then by point index, by the group.  The indices of one buffer are distinct, so every rank
// names one pair and the choice among equal values never depends on the gather order.
template <int GS, class CT>
__device__ void gpick(const Grp<GS>& q, const float* buf, const int* ib, int cnt, int s1, int s2, CT& C, float& o1,
                      float& o2, int& i1, int& i2)
{
    // tpk adjacent threads (one warp) rank one pair, each against every tpk-th pair, and add their counts:
    // small sets are ranked in about cnt / tpk dependent steps.  Every thread of the group runs the same
    // number of outer iterations, so the shuffles see whole warps.
    const int tpk = cnt * 8 <= GS ? 8 : (cnt * 4 <= GS ? 4 : (cnt * 2 <= GS ? 2 : 1));
    const int sub = q.t & (tpk - 1);
    for (int t0 = 0; t0 < cnt; t0 += GS / tpk) {
        const int t = t0 + q.t / tpk;
        const bool live = t < cnt;
        int r = 0;
        float v = 0.f;
        int iv = 0;
        if (live) {
            v = buf[t];
            iv = ib[t];
#pragma unroll 4
            for (int s = sub; s < cnt; s += tpk) {
                const float w2 = buf[s];
                r += (w2 < v) | ((w2 == v) & (ib[s] < iv));
            }
        }
        for (int o = 1; o < tpk; o <<= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, o);
        if (live && sub == 0) {
            if (r == s1) {
                C.pv1[q.g] = v;
                C.pi1[q.g] = iv;
            }
            if (r == s2) {
                C.pv2[q.g] = v;
                C.pi2[q.g] = iv;
            }
        }
    }
    q.sync();
    o1 = C.pv1[q.g];
    o2 = C.pv2[q.g];
    i1 = C.pi1[q.g];
    i2 = C.pi2[q.g];
    q.sync();
}

// Ranks s1 <= s2 among the pairs (buf, ib)[0..cnt), every value in [lo, hi], ordered like gpick, for
// sets too large for its all-pairs ranking: a 256-bucket histogram of the values (h2, 256 counters),
// one warp's scan locates the buckets of the two ranks, their few pairs move to (tb, ti) and gpick ranks
// them there.  Buckets are monotone in the value, so the rank of a pair is the count in lower buckets
// plus its rank within its own bucket.
constexpr int NB2 = 256;
static_assert(NB2 + 2 * CAP1H == NB, "D_P runs in the histogram area: NB2 counters, then CAP1H values and CAP1H indices");
// False, and nothing picked, where the values have no range or the ranks' buckets hold more pairs than (tb, ti).
template <int GS, class CT, int TCAP>
__device__ bool gpick_bins(const Grp<GS>& q, const float* buf, const int* ib, int cnt, int s1, int s2, float lo,
                           float hi, unsigned* h2, float* tb, int* ti, CT& C, float& o1, float& o2, int& i1,
                           int& i2)
{
    if (cnt <= 64) {
        gpick(q, buf, ib, cnt, s1, s2, C, o1, o2, i1, i2);
        return true;
    }
    if (!(lo < hi)) return false;
    float scale = __fdiv_rn((float)NB2, __fsub_rn(hi, lo));
    if (!(scale <= FLT_MAX)) scale = FLT_MAX;
    for (int b = q.t; b < NB2; b += GS) h2[b] = 0u;
    if (q.t == 0) C.gn[q.g] = 0;
    q.sync();
    auto bk = [&](float v) {
        const int b = __float2int_rz(__fmul_rn(__fsub_rn(v, lo), scale));
        return b < 0 ? 0 : (b > NB2 - 1 ? NB2 - 1 : b);
    };
    for (int t = q.t; t < cnt; t += GS) atomicAdd(&h2[bk(buf[t])], 1u);
    q.sync();
    if (q.t < 32) {
        constexpr int PER2 = NB2 / 32;
        const int lane = q.t;
        unsigned v[PER2];
        int own = 0;
#pragma unroll
        for (int k = 0; k < PER2; ++k) {
            v[k] = h2[lane * PER2 + k];
            own += (int)v[k];
        }
        int incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        int c = incl - own;
#pragma unroll
        for (int k = 0; k < PER2; ++k) {
            const int hk = (int)v[k];
            if (hk > 0) {
                if (c <= s1 && s1 < c + hk) {
                    C.f_b1[q.g] = lane * PER2 + k;
                    C.f_c1[q.g] = c;
                }
                if (c <= s2 && s2 < c + hk) {
                    C.f_b2[q.g] = lane * PER2 + k;
                    C.f_c2[q.g] = c;
                }
            }
            c += hk;
        }
    }
    q.sync();
    const int b1 = C.f_b1[q.g], c1 = C.f_c1[q.g], b2 = C.f_b2[q.g];
    const int n2 = C.f_c2[q.g] + (int)h2[b2] - c1;
    if (n2 > TCAP) return false;
    for (int t = q.t; t < cnt; t += GS) {
        const float v = buf[t];
        const int b = bk(v);
        if (b >= b1 && b <= b2) {
            const int pos = atomicAdd(&C.gn[q.g], 1);
            if (pos < TCAP) {
                tb[pos] = v;
                ti[pos] = ib[t];
            }
        }
    }
    q.sync();
    gpick(q, tb, ti, n2, s1 - c1, s2 - c1, C, o1, o2, i1, i2);
    return true;
}

// The same for every set: the whole of it is ranked where gpick_bins picks nothing.
template <int GS, class CT, int TCAP = CAP>
__device__ __forceinline__ void gpick_wide(const Grp<GS>& q, const float* buf, const int* ib, int cnt, int s1, int s2,
                                           float lo, float hi, unsigned* h2, float* tb, int* ti, CT& C, float& o1,
                                           float& o2, int& i1, int& i2)
{
    if (!gpick_bins<GS, CT, TCAP>(q, buf, ib, cnt, s1, s2, lo, hi, h2, tb, ti, C, o1, o2, i1, i2))
        gpick(q, buf, ib, cnt, s1, s2, C, o1, o2, i1, i2);
}

// Generic exact selection of rank q1 over one direction's values f(0..L-1),
// all in [lo, hi], by iterated bucketing (the fallback path); hist, buf and ibuf are the
// direction's own areas.  Returns the value and its point index.  One rank at a time: its bucket narrows every
// round, where the run of two ranks in two groups of equal values would never shrink.  Rank q2 >= q1 comes along
// where it lies in the group that ends the search (returns true).
template <int GS, class CT, class F, int FBN = FB_NB, int FBC = FB_CAP>
__device__ __noinline__ bool gselect1(const Grp<GS>& q, F f, int L, int q1, int q2, float lo, float hi, unsigned* hist, float* buf,
                         int* ibuf, CT& C, float& v1, int& i1, float& v2, int& i2, int* err)
{
    int below = 0, left = L;   // values below the candidates, and candidates
    for (int iter = 0; iter < 24; ++iter) {
        if (!(lo < hi)) {
            // every remaining candidate equals lo: the rank holds that value, taken at the smallest point index
            // that holds it (-1 if none does: values that are not numbers)
            if (q.t == 0) C.gi[q.g] = 0x7FFFFFFF;
            q.sync();
            for (int i = q.t; i < L; i += GS) {
                if (f(i) == lo) {
                    atomicMin(&C.gi[q.g], i);
                    break;
                }
            }
            q.sync();
            v1 = lo;
            i1 = C.gi[q.g] == 0x7FFFFFFF ? -1 : C.gi[q.g];
            v2 = v1;
            i2 = i1;
            q.sync();
            return q2 - below < left;
        }
        float scale = __fdiv_rn((float)FBN, __fsub_rn(hi, lo));
        if (!(scale <= FLT_MAX)) scale = FLT_MAX;
        for (int b = q.t; b < FBN / 4; b += GS) reinterpret_cast<uint4*>(hist)[b] = make_uint4(0u, 0u, 0u, 0u);
        q.sync();
        for (int i = q.t; i < L; i += GS) {
            const float a = f(i);
            if (a >= lo && a <= hi) atomicAdd(&hist[bucket<FBN>(a, lo, scale)], 1u);
        }
        q.sync();
        int b1, c1, b2, c2;
        gfind<GS, CT, FBN>(q, hist, q1 - below, q1 - below, C, b1, c1, b2, c2);
        const int cnt = (int)hist[b1];
        if (q.t == 0) C.gn[q.g] = 0;
        q.sync();
        if (cnt <= FBC) {
            for (int i = q.t; i < L; i += GS) {
                const float a = f(i);
                if (a >= lo && a <= hi) {
                    if (bucket<FBN>(a, lo, scale) == b1) {
                        const int pos = atomicAdd(&C.gn[q.g], 1);
                        if (pos < FBC) {
                            buf[pos] = a;
                            ibuf[pos] = i;
                        }
                    }
                }
            }
            q.sync();
            const int r1 = q1 - below - c1, r2 = q2 - below - c1;
            gpick(q, buf, ibuf, cnt, r1, r2 < cnt ? r2 : r1, C, v1, v2, i1, i2);
            return r2 < cnt;
        }
        float nlo = FLT_MAX, nhi = -FLT_MAX;
        for (int i = q.t; i < L; i += GS) {
            const float a = f(i);
            if (a >= lo && a <= hi) {
                if (bucket<FBN>(a, lo, scale) == b1) {
                    nlo = fminf(nlo, a);
                    nhi = fmaxf(nhi, a);
                }
            }
        }
        gminmax(q, nlo, nhi, C, lo, hi);
        below += c1;
        left = cnt;
    }
    if (q.t == 0) atomicOr(err, ERR_SELECT_ITER);
    v1 = v2 = __int_as_float(0x7FC00000);
    i1 = i2 = -1;
    return true;
}

// Two ranks q1 <= q2 by gselect1.
template <int GS, class CT, class F>
__device__ __forceinline__ void gselect(const Grp<GS>& q, F f, int L, int q1, int q2, float lo, float hi, unsigned* hist,
                                        float* buf, int* ibuf, CT& C, float& v1, float& v2, int& i1, int& i2, int* err)
{
    if (gselect1(q, f, L, q1, q2, lo, hi, hist, buf, ibuf, C, v1, i1, v2, i2, err)) return;
    float w;
    int j;
    gselect1(q, f, L, q2, q2, lo, hi, hist, buf, ibuf, C, v2, i2, w, j, err);
}

// One direction's keys held in an array: shared memory (resident keys) or device memory (keys formed
// by launch_pdap_keys when they do not fit shared memory).
struct KeysArray {
    const float* y;
    __device__ __forceinline__ float get(int i) const { return y[i]; }
    __device__ __forceinline__ float4 get4(int i) const { return *reinterpret_cast<const float4*>(y + i); }
};

// D_P's MAD from the gathered runs L, R (keys B1[0..cnt1), point indices I1) once the median m is known:
// the deviations replace the keys in place and the ranks s1 <= s2 among them are picked (gpick_wide, with
// h2 and the TCAP pairs tb / ti as scratch).  Every key between the runs lies in (max L, min R) and every
// key outside them below min L or above max R, so the picks are the MAD ranks of all keys when the
// deviations those bounds allow do not cross them; returns whether they do not (else nothing is picked
// for sure and the caller takes the |y - med| histogram pass).
template <int GS, int TCAP, class CT>
__device__ bool mad_from_runs(const Grp<GS>& q, float* B1, int* I1, int cnt1, int s1, int s2, float m, unsigned* h2,
                              float* tb, int* ti, CT& C, float& p1, float& p2, int& ip1, int& ip2)
{
    float lmin = FLT_MAX, lmax = -FLT_MAX, rmin = FLT_MAX, rmax = -FLT_MAX;
    for (int t = q.t; t < cnt1; t += GS) {
        const float v = B1[t];
        if (v < m) {   // L keys lie below m1 <= m, R keys above m2 >= m
            lmin = fminf(lmin, v);
            lmax = fmaxf(lmax, v);
        } else {
            rmin = fminf(rmin, v);
            rmax = fmaxf(rmax, v);
        }
        B1[t] = fabsf(__fsub_rn(v, m));
    }
    gminmax2(q, lmin, lmax, rmin, rmax, C);
    const float la = lmin, lb = lmax, ra = rmin, rb = rmax;
    if (!(lb > -FLT_MAX && ra < FLT_MAX && s1 >= 0 && s2 < cnt1)) return false;
    const float inner = fmaxf(__fsub_rn(m, lb), __fsub_rn(ra, m));
    const float outer = fminf(__fsub_rn(m, la), __fsub_rn(rb, m));
    gpick_wide<GS, CT, TCAP>(q, B1, I1, cnt1, s1, s2, fminf(__fsub_rn(m, lb), __fsub_rn(ra, m)),
                             fmaxf(__fsub_rn(m, la), __fsub_rn(rb, m)), h2, tb, ti, C, p1, p2, ip1, ip2);
    return inner <= p1 && outer >= p2;
}

// The points a selection kernel picked for one direction are written into the direction's result cell in
// place of its depth, which k_pdap_finish then forms from them: the points of the median ranks (im1, im2)
// and of the MAD or MAD_+ ranks (ip1, ip2); -1 where a selection failed (its error flag is set), and
// ip1 = ip2 = NOPOS for D_AP when no key lies above the median (MAD_+ = 0).  Two 8-byte stores: a result
// cell is 8-byte aligned.
constexpr int NOPOS = -2;
__device__ __forceinline__ void put_picks(ResDev* cell, int im1, int im2, int ip1, int ip2)
{
    int2* c = reinterpret_cast<int2*>(cell);
    c[0] = make_int2(im1, im2);
    c[1] = make_int2(ip1, ip2);
}

}  // namespace
}  // namespace rrs
