// Filters of the fold: upper bounds on the ln P of many cells at once, from
// tables indexed by slot.
//
// A fold has n_phi x n_D cells per period and one addition per (cell, event)
// at the least; nearly every cell is far below the best one.  The filters
// bound cells from a few bytes per event, several phases and durations per
// lane, and only the cells they do not rule out go on to the full FP32 screen
// (fold's queue A) and from there to the exact evaluation.
//
// Bounds.  With y_k = Delta_k / s_k, v_k = 1 / s_k^2 and the bound of the
// screen (ln P <= S_L + 1/2 - q / (2 (1 + x_max)), q = sum y_k^2 -
// (sum Delta_k v_k)^2 / sum v_k), for any beta <= 1 / (2 (1 + x_max)):
//   ln P <= 1/2 + sum_k (l_k - beta y_k^2) + beta (sum_k Delta_k v_k)^2 / sum_k v_k.
// x_max <= max v / sum v, so beta is allowed when sum v >= max v 2 beta / (1 - 2 beta).
// Two facts keep this a sum over events of per-slot numbers:
//  (split)  (A1 + A2)^2 / (V1 + V2) <= A1^2 / V1 + A2^2 / V2 for V > 0 (Cauchy):
//           an event that may or may not take part (its slot touches both a
//           valid and an invalid interval) adds at most its gain l_k alone;
//  (error)  an event whose Delta v is only known to within e adds
//           beta e^2 / (tau v_k) to the sum when the quadratic term takes
//           beta / (1 - tau): the same inequality on (1 - tau) v and tau v.
// Per slot and duration the tables hold, for every event position the exact
// path can have while its walk position is in the slot (a margin of 2^-14 slot
// on either side covers the walk's error):
//   L    the largest gain l (0: no event);
//   S    a chord of Delta v over the slot (value and slope), the smallest v and
//        the largest l - beta y^2 + error term with beta = FILTER_BETA_A;
//   gB   the last with beta = FILTER_BETA_B;
// with Delta v in units of sqrt(max v) and v in units of max v of the duration.
// From these, for several phases at once (neighbouring phases are at most one
// slot apart at every epoch):
//   Q    over four slots: the largest and smallest Delta v, the smallest v, the
//        largest gB (four phases of one duration);
//   G    over eight slots: the largest L (eight phases of up to eight durations).
// S and Q are packed as the high halves of two words whose low halves hold
// another BF16 number: the word itself is read as the FP32 value of the high
// half, and its rounding direction is chosen with the low half in place.
// G and L are FP32, and so are all sums (G as FP16 with FP16 sums: 1 to 4 % faster
// on the folds of 10 to 20 durations, but 2^-11 of the sum looser per event, and
// a gain above 65 504 passed everything).
// Q and G are stored by slot modulo 4 and 8, so that the lanes of a warp, on
// consecutive groups of phases, read consecutive entries.
//
// Which filter serves a period depends on K = span / P, the epochs of a cell.
// Fractions of cells passed at the final threshold, two-minute light curves of
// 19 440 / 136 080 epochs (synthetic, 10 / 20 durations): G 0.5-1.5 % at K <= 4
// and 9 / 3 % at K = 5; Q 1.4 / 0.4 % at K = 6, 1.3 / 0.3 % at 8, 12 / 3 % at
// 16; the cell bound of S 0.04 % / 0.002 % at 24, 0.9 / 0.02 % at 50.
#pragma once

#include <cuda_fp16.h>

#include "fold.cuh"

namespace nu {

#define FILTER_BETA_A 0.465f    // x_max <= 1/13.3
#define FILTER_BETA_B 0.38f     // x_max <= 1/3.2
#define FILTER_TAU 0.125f
#define FILTER_K_QUAD 5.5f   // epochs per cell from which Q bounds better than G
#define FILTER_K_CELL 22.0f  // and S better than Q
#define FILTER_K_A 16.5f        // and beta A is allowed (with a margin for holes)
#define FILTER_K_MID 3.8f    // groups that G passes are bounded by Q next
#define FILTER_K_MAX 4000.0f    // FP32 sums: K 2^-24 stays below the tables' slack
// margin of the tables in walk units (2^-40 slot); a period's band half-width
// delta (16 times the walk's error) must not exceed 16 times this
#define FILTER_MARGIN (1ull << 26)

// ------------------------------------------------------------------ tables
// The curve of table row entry o (segs: the batch's curves, else the one
// curve) and the entry's duration and slot.
struct FilterSlot {
    int seg, d, s;
};
__device__ __forceinline__ bool filter_slot(const FoldSeg* __restrict__ segs,
                                            const FoldSeg& one, int n_seg, int n_D, int64_t o,
                                            FilterSlot& fs, FoldSeg& sg) {
    fs.seg = 0;
    if (segs) {
        int lo = 0, hi = n_seg;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (segs[mid].tab_off <= o) lo = mid; else hi = mid;
        }
        fs.seg = lo;
        sg = segs[lo];
    } else {
        sg = one;
    }
    const int64_t ns = filter_slots(sg.n_slots);
    const int64_t r = o - sg.tab_off;
    if (r < 0 || r >= ns * n_D) return false;
    fs.d = (int)(r / ns);
    fs.s = (int)(r - (int64_t)fs.d * ns);
    return true;
}

// A word whose FP32 value is at least (up) or at most (!up) x, with the BF16
// bits lo in its low half (x finite or +inf; a word of magnitude below 2^-126
// stands for 0).
__device__ __forceinline__ unsigned pack_hi(float x, unsigned lo, bool up) {
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu, sign = b & 0x80000000u;
    unsigned h = m >> 16;
    const bool away = (sign == 0u) == up;              // the magnitude may grow, not shrink
    if (away) {
        if (((h << 16) | lo) < m) ++h;
        if (h >= 0x7f80u) return sign | 0x7f800000u;   // infinite: the low half must be 0
    } else if (((h << 16) | lo) > m && h > 0u) {
        --h;
    }
    return sign | (h << 16) | lo;
}
// The word nearest to x (to 2^-8 relative) with lo in its low half.
__device__ __forceinline__ unsigned pack_near(float x, unsigned lo) {
    const unsigned b = __float_as_uint(x);
    unsigned h = b >> 16;
    const int d = (int)(b & 0xffffu) - (int)lo;        // truncated error
    if (d > 0x8000) ++h;
    else if (d < -0x8000 && (h & 0x7fffu) != 0u) --h;
    return (h << 16) | lo;
}
__device__ __forceinline__ unsigned bf16_bits_ru(float x) {
    const unsigned b = __float_as_uint(x);
    if (b >> 31) return b >> 16;                       // towards zero
    const unsigned h = (b + 0xffffu) >> 16;
    return h > 0x7f80u ? 0x7f80u : h;
}
__device__ __forceinline__ unsigned bf16_bits_rn(float x) {
    const unsigned b = __float_as_uint(x);
    return (b + 0x7fffu + ((b >> 16) & 1u)) >> 16;
}

// The part of one valid interval that a slot's events can lie on: the values
// at its two ends (Delta v in units of sqrt(max v)) and bounds inside.
struct Portion {
    float h0, h1;      // Delta v at the ends
    float dev;         // |Delta v - chord| inside
    float v;           // smallest v / max v
    float l;           // largest gain
    float y0, y1, g0, l0, l1, ydev;
};
// Delta, sigma, gain at the ends of the part; rs = 1 / sqrt(max v).
__device__ __forceinline__ Portion portion(float d0, float s0, float l0, float d1, float s1,
                                           float l1, float rs) {
    Portion p;
    const float i0 = 1.f / s0, i1 = 1.f / s1;
    const float sm = fminf(s0, s1), im = 1.f / sm;
    const float dd = fabsf(d1 - d0), ds = fabsf(s1 - s0), dm = fmaxf(fabsf(d0), fabsf(d1));
    p.y0 = d0 * i0;
    p.y1 = d1 * i1;
    p.h0 = p.y0 * (i0 * rs);
    p.h1 = p.y1 * (i1 * rs);
    // |f - chord| <= max |f''| / 8 on the unit interval, for f = d / s^2 and d / s
    const float e = ds * im;
    p.dev = (0.5f * dd * e + 0.75f * dm * e * e) * im * (im * rs) * 1.01f;
    p.ydev = (0.25f * dd * e + 0.25f * dm * e * e) * im * 1.01f;
    const float sx = fmaxf(s0, s1);
    p.v = (1.f / sx) * (1.f / sx) * (rs * rs) * (1.f - 4e-6f);
    p.l0 = l0;
    p.l1 = l1;
    p.l = fmaxf(l0, l1);
    p.g0 = 0.f;
    return p;
}
// Largest l - beta y^2 on the part (the quadratic's chord deviation is at
// most beta (y1 - y0)^2 / 4), with slack for the FP32 arithmetic.
__device__ __forceinline__ float portion_g(const Portion& p, float beta) {
    const float a = p.l0 - beta * p.y0 * p.y0, b = p.l1 - beta * p.y1 * p.y1;
    const float ym = fmaxf(fabsf(p.y0), fabsf(p.y1));
    const float dy = p.y1 - p.y0;
    return fmaxf(a, b) + beta * (0.25f * dy * dy + p.ydev * (2.f * ym + p.ydev)) * 1.0001f +
           2e-6f * (fabsf(p.l0) + fabsf(p.l1) + ym * ym);
}

// Whether the interval between two slot records is outside what is bounded.
__device__ __forceinline__ bool slot_odd(const Node4<float>& a, const Node4<float>& b) {
    return !(a.s >= 1e-12f && a.s <= 1e12f) || !(b.s >= 1e-12f && b.s <= 1e12f) ||
           !(a.s <= 3.f * b.s) || !(b.s <= 3.f * a.s) || !(fabsf(a.d) <= 1e8f * a.s) ||
           !(fabsf(b.d) <= 1e8f * b.s) || !(fabsf(a.l) <= 1e20f) || !(fabsf(b.l) <= 1e20f);
}
// L of a slot: its largest gain lmax with room for rounding, +inf where it is not
// bounded.
__device__ __forceinline__ float bounded_gain(float lmax, bool odd) {
    const float l = fmaxf(lmax * 1.000001f, 1e-30f);
    return odd || !(l < 1e30f) ? INFINITY : l;
}
__device__ __forceinline__ float slot_gain(const Node4<float>& a, const Node4<float>& b) {
    return bounded_gain(fmaxf(a.l, b.l), slot_odd(a, b));
}

// Writes the entries of one slot.  ok: every event of the slot is on a valid
// interval (chord from zA to zB, within e; the smallest v; the largest gA,
// gB); maybe: some are, some are not (their gains lmax count); odd: not bounded.
__device__ __forceinline__ void write_slot(const FilterTab& tab, int64_t o, int64_t so,
                                           bool any, bool mixed, bool odd, float zA, float zB, float e, float v,
                                           float gA, float gB, float lmax) {
    const float tiny = 1e-30f;
    if (!tab.S) {                       // the gains alone
        tab.L[o] = any ? bounded_gain(lmax, odd) : 0.f;
        return;
    }
    float z0 = 0.f, dz = 0.f, vv = 0.f, a = 0.f, b = 0.f, l = 0.f, zmx = 0.f, zmn = 0.f;
    if (any) {
        l = fmaxf(lmax * 1.000001f, tiny);
        if (mixed || odd) {
            a = b = l;
        } else {
            z0 = zA;
            dz = zB - zA;
            // packing (2^-8 of value and slope) and the rounding of the sums
            e += 0.0079f * (fabsf(z0) + fabsf(dz));
            zmx = fmaxf(zA, zB) + e;
            zmn = fminf(zA, zB) - e;
            vv = v;
            const float q = e * e / (FILTER_TAU * v) * 1.001f;
            a = fmaxf(gA, tiny) + FILTER_BETA_A * q;
            b = fmaxf(gB, tiny) + FILTER_BETA_B * q;
            // outside what the packed numbers hold, or no number at all
            if (!(fabsf(z0) < 3e4f) || !(fabsf(dz) < 3e4f) || !(zmx < 6e4f) || !(zmn > -6e4f) ||
                !(vv > 1e-30f) || !(a < 1e30f) || !(b < 1e30f))
                odd = true;
        }
        if (odd || !(l < 1e30f)) {
            z0 = dz = vv = zmx = zmn = 0.f;
            a = b = l = INFINITY;
        }
    }
    tab.S[so] = make_uint2(pack_near(z0, bf16_bits_rn(dz)), pack_hi(vv, bf16_bits_ru(a), false));
    tab.gB[o] = b;
    tab.L[o] = l;
    const __half hx = __float2half_ru(zmx), hn = __float2half_rd(zmn);
    tab.Z[o] = (unsigned)__half_as_ushort(hx) << 16 | (unsigned)__half_as_ushort(hn);
}

// max 1/s^2 of each duration's valid intervals (vmax zero on entry)
__global__ void k_filter_vmax(const ScreenRec* __restrict__ screen,
                              const Node4<float>* __restrict__ rec,
                              const FoldSeg* __restrict__ segs, FoldSeg one, int n_D,
                              unsigned* __restrict__ vmax) {
    const int seg = blockIdx.x / n_D, d = blockIdx.x - seg * n_D;
    const FoldSeg sg = segs ? segs[seg] : one;
    float m = 0.f;
    if (sg.use_slots) {
        const Node4<float>* r = rec + sg.rec_off + (int64_t)d * sg.n_slots;
        for (int64_t i = blockIdx.y * (int64_t)blockDim.x + threadIdx.x; i < sg.n_slots;
             i += (int64_t)gridDim.y * blockDim.x) {
            const float s = r[i].s;
            if (s >= 1e-12f && s <= 1e12f) m = fmaxf(m, 1.f / (s * s));
        }
    } else if (sg.screen) {
        const ScreenRec* r = screen + sg.s_off * n_D + (int64_t)d * sg.n_t0;
        for (int64_t i = blockIdx.y * (int64_t)blockDim.x + threadIdx.x; i < sg.n_t0;
             i += (int64_t)gridDim.y * blockDim.x) {
            const float s = r[i].s, s1 = s + r[i].ds;
            if (s < INFINITY && !r[i].flags) m = fmaxf(m, fmaxf(1.f / (s * s), 1.f / (s1 * s1)));
        }
    }
    m *= 1.00001f;
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.f && m < INFINITY)
        atomicMax(vmax + blockIdx.x, __float_as_uint(m));
}

// S and Q hold the durations in pairs, two entries per slot: entry of duration
// d at position s (a slot, or its place modulo 4).
__device__ __forceinline__ int64_t filter_pair(const FoldSeg& sg, int n_D, int d, int64_t s) {
    const int64_t ns = filter_slots(sg.n_slots);
    return sg.pair_off + ((int64_t)(d >> 1) * ns + s) * 2 + (d & 1);
}

// L, S, gB and Z of every (duration, slot).  Grids of the exact paths: from
// the screening records and epoch positions (the last epoch's interval is
// invalid, so the slot that holds it only counts its gains).  Slot path: an
// event in slot s interpolates the records of s and s + 1, nothing else.
__global__ void k_filter_slots(const ScreenRec* __restrict__ screen,
                               const ulonglong2* __restrict__ vpair,
                               const int* __restrict__ bucket,
                               const Node4<float>* __restrict__ rec,
                               const FoldSeg* __restrict__ segs, FoldSeg one, int n_seg, int n_D,
                               int64_t n_entries, FilterTab tab) {
    const int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (o >= n_entries) return;
    FilterSlot fs;
    FoldSeg sg;
    if (!filter_slot(segs, one, n_seg, n_D, o, fs, sg)) return;
    const int64_t so = filter_pair(sg, n_D, fs.d, fs.s);
    if (tab.S && fs.d == n_D - 1 && (n_D & 1))       // the other half of the last pair
        tab.S[so + 1] = make_uint2(0u, 0u);
    const float vm = tab.S ? __uint_as_float(tab.vmax[fs.seg * n_D + fs.d]) : 0.f;
    const float rs = vm > 0.f ? 1.f / sqrtf(vm) : 0.f;
    bool any = false, none = false, odd = false;
    float zA = 0.f, zB = 0.f, e = 0.f, v = INFINITY, gA = -INFINITY, gB = -INFINITY;
    float lmax = -INFINITY;
    if (sg.use_slots) {
        if (fs.s + 1 < sg.n_slots) {
            const Node4<float>* r = rec + sg.rec_off + (int64_t)fs.d * sg.n_slots + fs.s;
            const Node4<float> a = r[0], b = r[1];
            if (!isnan(a.s) && !isnan(b.s)) {
                any = true;
                odd = slot_odd(a, b);
                if (!odd) {
                    const Portion p = portion(a.d, a.s, a.l, b.d, b.s, b.l, rs);
                    zA = p.h0;
                    zB = p.h1;
                    e = p.dev;
                    v = p.v;
                    gA = portion_g(p, FILTER_BETA_A);
                    gB = portion_g(p, FILTER_BETA_B);
                    lmax = p.l;
                }
            }
        }
        // The last epoch may lie up to 1e-3 slot before its slot: positions past it
        // on the interval that ends there have no event, and a group's walk may
        // reach them while its first phase has not (only the gains count then).
        const bool past = ((unsigned long long)fs.s + 1ull) << 40 > sg.ulast + 1ull;
        write_slot(tab, o, so, any, past, odd, zA, zB, e, v, gA, gB, lmax);
        return;
    }
    if (!sg.screen) return;
    const ulonglong2* vp = vpair + sg.s_off;
    const ScreenRec* row = screen + sg.s_off * n_D + (int64_t)fs.d * sg.n_t0;
    const int* bk = bucket + sg.bucket_off;
    const unsigned long long at = (unsigned long long)fs.s << 40, one40 = 1ull << 40;
    const unsigned long long lo = at > FILTER_MARGIN ? at - FILTER_MARGIN : 0ull;
    const unsigned long long hi = at + one40 + FILTER_MARGIN;
    int64_t i = (int64_t)bk[fs.s < sg.n_bucket ? fs.s : sg.n_bucket - 1] - 1;
    if (i < 0) i = 0;
    while (i > 0 && vp[i].x > lo) --i;
    while (i + 1 < sg.n_t0 && vp[i + 1].x <= lo) ++i;
    const int64_t i0 = i;
    // slot coordinate of a position (the slot is [0, 1))
    auto coord = [&](unsigned long long p) {
        const long long r = (long long)(p - at);
        return (float)(int)max(min(r >> 16, 0x3fffffffll), -0x3fffffffll) * 5.9604645e-08f;
    };
    const float bm = (float)FILTER_MARGIN * 9.094947e-13f;
    float slope = 0.f;
    for (i = i0; i < sg.n_t0 && vp[i].x < hi; ++i) {
        const ScreenRec r = row[i];
        if (isnan(r.s)) {
            none = true;
            continue;
        }
        any = true;
        if (r.flags) {
            odd = true;
            break;
        }
        const float p = coord(vp[i].x), q = coord(vp[i].y);
        const float iw = 1.f / (q - p);
        const float x0 = fmaxf(p, -bm), x1 = fminf(q, 1.f + bm);
        const float w0 = fmaxf((x0 - p) * iw, 0.f), w1 = fminf((x1 - p) * iw, 1.f);
        const Portion pt = portion(fmaf(w0, r.dd, r.d), fmaf(w0, r.ds, r.s),
                                   fmaf(w0, r.dl, r.l), fmaf(w1, r.dd, r.d),
                                   fmaf(w1, r.ds, r.s), fmaf(w1, r.dl, r.l), rs);
        const Portion fl = portion(r.d, r.s, r.l, r.d + r.dd, r.s + r.ds, r.l + r.dl, rs);
        v = fminf(v, pt.v);
        gA = fmaxf(gA, portion_g(pt, FILTER_BETA_A));
        gB = fmaxf(gB, portion_g(pt, FILTER_BETA_B));
        lmax = fmaxf(lmax, pt.l + 2e-6f * (fabsf(r.l) + fabsf(r.dl)));
        e = fmaxf(e, pt.dev);
        slope = fmaxf(slope, (fabsf(fl.h1 - fl.h0) + 8.f * fl.dev) * iw);
        if (p <= 0.f || i == i0) {            // the last interval that starts at or before s
            const float w = fminf(fmaxf(-p * iw, 0.f), 1.f);
            const float s = fmaf(w, r.ds, r.s);
            zA = fmaf(w, r.dd, r.d) / (s * s) * rs;
        }
        const float w = fminf(fmaxf((1.f - p) * iw, 0.f), 1.f);
        const float s = fmaf(w, r.ds, r.s);
        if (p < 1.f) zB = fmaf(w, r.dd, r.d) / (s * s) * rs;
    }
    if (any && !odd && !none) {
        // the chord against the values at the knots inside the slot
        float dev = 0.f;
        for (i = i0; i < sg.n_t0 && vp[i].x < hi; ++i) {
            const ScreenRec r = row[i];
            const float p = coord(vp[i].x);
            if (p > 0.f && p < 1.f)
                dev = fmaxf(dev, fabsf(r.d / (r.s * r.s) * rs - fmaf(p, zB - zA, zA)));
            const float q = coord(vp[i].y);
            if (q > 0.f && q < 1.f) {
                const float s = r.s + r.ds;
                dev = fmaxf(dev, fabsf((r.d + r.dd) / (s * s) * rs - fmaf(q, zB - zA, zA)));
            }
        }
        e += dev + 2.f * bm * (slope + fabsf(zB - zA));
    }
    write_slot(tab, o, so, any, none, odd, zA, zB, e, v, gA, gB, lmax);
}

// Q and G from the slot entries.
__global__ void k_filter_groups(const FoldSeg* __restrict__ segs, FoldSeg one, int n_seg,
                                int n_D, int64_t n_entries, FilterTab tab) {
    const int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (o >= n_entries) return;
    FilterSlot fs;
    FoldSeg sg;
    if (!filter_slot(segs, one, n_seg, n_D, o, fs, sg)) return;
    if (!sg.use_slots && !sg.screen) return;
    const int ns = (int)filter_slots(sg.n_slots);
    const int64_t s0 = filter_pair(sg, n_D, fs.d, 0);
    float mx = -INFINITY, mn = INFINITY, v = INFINITY, g = 0.f, l = 0.f;
    for (int w = 0; w < 8; ++w) {
        if (fs.s + w >= ns) {
            if (w < 4) {
                mx = fmaxf(mx, 0.f);
                mn = fminf(mn, 0.f);
                v = 0.f;
            }
            break;
        }
        l = fmaxf(l, tab.L[o + w]);
        if (w < 4 && tab.S) {
            const unsigned z = tab.Z[o + w];
            mx = fmaxf(mx, __half2float(__ushort_as_half((unsigned short)(z >> 16))));
            mn = fminf(mn, __half2float(__ushort_as_half((unsigned short)(z & 0xffffu))));
            v = fminf(v, __uint_as_float(tab.S[s0 + 2 * (int64_t)(fs.s + w)].y & 0xffff0000u));
            g = fmaxf(g, tab.gB[o + w]);
        }
    }
    // (-mn and mx: both rounded up; the low half of a word holds the other
    // number as BF16)
    if (tab.S) {
        const int64_t qo =
            filter_pair(sg, n_D, fs.d, (int64_t)(fs.s & 3) * (ns >> 2) + (fs.s >> 2));
        tab.Q[qo] = make_uint2(pack_hi(mx, bf16_bits_ru(-mn), true),
                               pack_hi(v, bf16_bits_ru(g), false));
        if (fs.d == n_D - 1 && (n_D & 1)) tab.Q[qo + 1] = make_uint2(0u, 0u);
    }
    const int gi = fs.d >> 3, W = filter_width(n_D, gi), c = fs.d & 7;
    float* G = tab.G + sg.g_off + (int64_t)gi * 8 * ns +
               ((int64_t)(fs.s & 7) * (ns >> 3) + (fs.s >> 3)) * W;
    G[c] = l;
    if (fs.d == n_D - 1)
        for (int q = c + 1; q < W; ++q) G[q] = 0.f;
}

// ------------------------------------------------------------------ walks
// One curve's tables.
struct FilterView {
    const uint2* S;
    const float* gB;
    const float* L;
    const uint2* Q;
    const float* G;
    int ns;
};
__device__ __forceinline__ FilterView filter_view(const FilterTab& tab, const FoldSeg& sg) {
    FilterView v;
    v.S = tab.S ? tab.S + sg.pair_off : nullptr;
    v.Q = tab.S ? tab.Q + sg.pair_off : nullptr;
    v.gB = tab.S ? tab.gB + sg.tab_off : nullptr;
    v.L = tab.L + sg.tab_off;
    v.G = tab.G ? tab.G + sg.g_off : nullptr;
    v.ns = (int)filter_slots(sg.n_slots);
    return v;
}

enum { FILTER_NONE = 0, FILTER_GAIN = 1, FILTER_QUAD = 2, FILTER_CELL = 3, FILTER_LONE = 4 };

// One period's walk: epochs at u0 + k ustep < uend, u0 = j uph for phase j, in
// 2^-40 slots (2^32 <= ustep < 2^60, uend < 2^62: no position wraps).
struct FilterPeriod {
    unsigned long long ustep, uph, uend;
    int64_t n_phi;
    float K;              // at least the epochs of a cell
    int mode;
};
// Cells per lane of an item's nw warps up to which every cell is screened.  The
// filters start from a threshold that a few cells' screens give: three walks in
// a row of one and of eight lanes, and one of the filter, however few the cells.
// Long walks of few cells lose most: 10 000 periods uniform in frequency of
// 100 000 epochs, one duration, 8.7 -> 3.6 ms mixed and 8.7 -> 3.9 FP64; 3 500 of
// 19 440 x 10 linear, FP64, 1.63 -> 1.33.  Two or eight warps: 6 / 9 / 14 cells
// 2.10 / 1.88 / 1.99 ms on 3 500 of 19 440 x 10 uniform in frequency; one warp: 9 /
// 20 / 45 cells 86.1 / 81.6 / 90.0 ms on 1 000 curves of 2 880 x 4 000 periods.
// Where the screen searches the epochs' positions (!placed) it costs more, and only
// long walks are worth it.  All / none up to 9 cells: 20 000 periods of 19 440 x 10,
// FP64 (K to 135), 3.61 / 3.76 ms; 1 630 of 17 000 x 11, mixed (K 89), 1.36 / 1.44; but
// 2 026 uniform in frequency of 6 000 x 13, mixed (K 38), 1.22 / 1.15, and 12 586 of
// 3 200 x 11, FP64 (K 23), 1.74 / 1.63; one warp, 60 000 of 9 000 x 1, FP64 (K 13 to
// 43), 20 / 7 cells 4.76 / 4.07.
__device__ __forceinline__ int filter_rounds(int nw, bool placed, float K) {
    return !placed && K < 40.f ? 4 : (nw == 1 ? 20 : 9);
}
// (n_cells < 2^31: the filters count groups in 32 bits)
__device__ __forceinline__ int filter_mode(const FilterTab& tab, unsigned long long ustep,
                                           float K, int64_t n_cells, int nw, bool placed) {
    if (n_cells <= filter_rounds(nw, placed, K) * 32 * nw) return FILTER_NONE;
    if (!tab.L || ustep < (1ull << 32) || ustep >= (1ull << 60) || !(K < FILTER_K_MAX) ||
        n_cells >= 0x7fff0000LL)
        return FILTER_NONE;
    if (!tab.G) return FILTER_LONE;
    if (K < FILTER_K_QUAD) return FILTER_GAIN;
    // (without S and Q the cells one by one, by their gains; 19 440 epochs x 12
    // durations x 3 000 periods, FP64: 1.69 ms, 4.7 in groups of eight)
    if (!tab.S) return FILTER_LONE;
    return K < FILTER_K_CELL ? FILTER_QUAD : FILTER_CELL;
}

__device__ __forceinline__ float filter_weight(unsigned long long u) {
    return __uint_as_float(0x3f800000u | (unsigned)((u >> 17) & 0x7fffffu)) - 1.0f;
}

// Upper bound from the sums (Delta v, v, l - beta y^2): +inf where beta is not
// allowed (or nothing is known), -inf for a cell without an event.  c covers
// the rounding of the sums.
__device__ __forceinline__ float filter_bound(float sd, float v, float g, float eff, float xlim,
                                              float c) {
    if (v < 1e-30f && g == 0.f) return -INFINITY;
    const float vl = v * (1.f - c);
    if (!(vl * xlim >= 1.00001f)) return INFINITY;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(vl));
    return fmaf(g, 1.f + c, 0.500001f) + eff * sd * sd * r * 1.00001f;
}

// Gain sums of two groups of eight phases, of W durations each (rows r0, r1, walks
// from u0, u1).  64 bytes in flight a lane, two epochs of both groups or one:
// the walks are short (two to five epochs), so that a round is mostly the latency
// of its loads.  Positions past the end, of either walk, add terms >= 0 (the empty
// last entry, or an event the cell does not have).
template <int W> struct __align__(W >= 4 ? 16 : 4 * W) FilterEntry {
    float l[W];
};
template <int W>
__device__ __forceinline__ void filter_gain(const float* __restrict__ g0,
                                            const float* __restrict__ g1, unsigned ns,
                                            unsigned long long u0, unsigned long long u1,
                                            unsigned long long ustep, unsigned long long uend,
                                            float (&a)[8], float (&b)[8]) {
    typedef FilterEntry<W> V;
    const V* __restrict__ r0 = reinterpret_cast<const V*>(g0);
    const V* __restrict__ r1 = reinterpret_cast<const V*>(g1);
    const unsigned n8 = ns >> 3, last = ns - 1u;
    auto at = [&](unsigned long long x) {
        const unsigned s = min((unsigned)(x >> 40), last);
        return (s & 7u) * n8 + (s >> 3);
    };
    auto add = [&](float (&c)[8], const V& v) {
#pragma unroll
        for (int i = 0; i < W; ++i) c[i] += v.l[i];
    };
    constexpr int E = W == 8 ? 1 : 2;
    for (; min(u0, u1) < uend; u0 += E * ustep, u1 += E * ustep) {
        const V x0 = r0[at(u0)], x1 = r1[at(u1)];
        if (E == 2) {
            const V y0 = r0[at(u0 + ustep)], y1 = r1[at(u1 + ustep)];
            add(a, x0);
            add(b, x1);
            add(a, y0);
            add(b, y1);
        } else {
            add(a, x0);
            add(b, x1);
        }
    }
}

// One cell by its gains, or by S.
__device__ __forceinline__ float filter_one_gain(const FilterView& f, int d,
                                                 unsigned long long u, const FilterPeriod& fp,
                                                 float c) {
    const unsigned last = (unsigned)f.ns - 1u;
    const float* __restrict__ r = f.L + (int64_t)d * f.ns;
    float l = 0.f;
    for (; u < fp.uend; u += 2ull * fp.ustep) {
        const float a = r[min((unsigned)(u >> 40), last)];
        const float b = r[min((unsigned)((u + fp.ustep) >> 40), last)];
        l += a + b;
    }
    return l > 0.f ? fmaf(l, 1.f + c, 0.500001f) : -INFINITY;
}
__device__ __forceinline__ float filter_one(const FilterView& f, int d, unsigned long long u,
                                            const FilterPeriod& fp, float c) {
    const unsigned last = (unsigned)f.ns - 1u;
    const uint2* __restrict__ r = f.S + (int64_t)(d >> 1) * f.ns * 2 + (d & 1);
    const float* __restrict__ b = f.gB + (int64_t)d * f.ns;
    const bool A = fp.K >= FILTER_K_A + 2.f;
    float sd = 0.f, v = 0.f, g = 0.f;
    for (; u < fp.uend; u += 2ull * fp.ustep) {
        const unsigned long long u2 = u + fp.ustep;
        const unsigned s = min((unsigned)(u >> 40), last);
        const unsigned s2 = u2 < fp.uend ? min((unsigned)(u2 >> 40), last) : last;
        const uint2 x = r[2 * (size_t)s], y = r[2 * (size_t)s2];
        const float gx = A ? __uint_as_float(x.y << 16) : b[s];
        const float gy = A ? __uint_as_float(y.y << 16) : b[s2];
        sd += fmaf(filter_weight(u), __uint_as_float(x.x << 16), __uint_as_float(x.x)) +
              fmaf(filter_weight(u2), __uint_as_float(y.x << 16), __uint_as_float(y.x));
        v += __uint_as_float(x.y) + __uint_as_float(y.y);
        g += gx + gy;
    }
    const float beta = A ? FILTER_BETA_A : FILTER_BETA_B;
    return filter_bound(sd, v, g, beta / (1.f - FILTER_TAU), 1.f / (2.f * beta) - 1.f, c);
}

// Per-warp shared queues of the filters: groups of phases that passed, and
// cells for the full screen (ni, nq, nc: their lengths).
#define FILTER_ITEMS 96
struct FilterQueues {
    uint2 item[FILTER_ITEMS + 32];   // (group index, duration)
    uint2 quad[40];        // (group of four phases, duration) between G and the cells
    uint2 cell[64];        // (phase, duration)
    int ni, nq, nc;
};
// An item's filter state, in shared memory; bfk is the threshold (a lower
// bound of the best ln P as an order-preserving key, may rise at any time).
struct FilterCtx {
    FilterView f;
    FilterPeriod fp;
    int n_D;
    unsigned bfk;
};

// Order-preserving unsigned key of a float (for a shared atomic max).
__device__ __forceinline__ unsigned fkey(float x) {
    const unsigned b = __float_as_uint(x);
    return (b >> 31) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_fkey(unsigned k) {
    return __uint_as_float((k >> 31) ? (k & 0x7fffffffu) : ~k);
}
__device__ __forceinline__ float filter_thr(const FilterCtx& x) {
    return from_fkey(*(const volatile unsigned*)&x.bfk);
}
__device__ __forceinline__ void filter_raise(FilterCtx& x, unsigned key) {
    if (key > *(volatile unsigned*)&x.bfk) atomicMax(&x.bfk, key);
}
// phases of one group, as a shift
__device__ __forceinline__ int filter_shift(int mode) {
    return mode == FILTER_GAIN ? 3 : (mode == FILTER_QUAD ? 2 : 0);
}
__device__ __forceinline__ float filter_slack(const FilterPeriod& fp) {
    return (fp.K + 8.f) * 1.1920929e-7f;
}

// Gain sums of the groups (q0, g0) and (q1, g1).
struct FilterGains {
    float a[8], b[8];
};
template <int W>
__device__ __forceinline__ void filter_gains(const FilterCtx& x, unsigned q0, int g0, unsigned q1,
                                             int g1, FilterGains& s) {
#pragma unroll
    for (int i = 0; i < 8; ++i) s.a[i] = s.b[i] = 0.f;
    const unsigned ns = (unsigned)x.f.ns;
    const unsigned long long uph8 = x.fp.uph << 3;
    filter_gain<W>(x.f.G + (int64_t)g0 * 8 * (int)ns, x.f.G + (int64_t)g1 * 8 * (int)ns, ns,
                   q0 * uph8, q1 * uph8, x.fp.ustep, x.fp.uend, s.a, s.b);
}
// Which of them reach the threshold: bit i is duration i of the first group,
// bit 16 + i of the second.
template <int W>
__device__ __forceinline__ unsigned filter_gain_pass(const FilterCtx& x, unsigned q0, int g0,
                                                     unsigned q1, int g1) {
    FilterGains s;
    filter_gains<W>(x, q0, g0, q1, g1, s);
    // (a sum of 0, no event, is below every entry)
    const float t = fmaxf((filter_thr(x) - 0.500002f) * (1.f - filter_slack(x.fp)), 5e-31f);
    unsigned pass = 0u;
#pragma unroll
    for (int i = 0; i < W; ++i)
        pass |= (s.a[i] >= t ? 1u << i : 0u) | (s.b[i] >= t ? 0x10000u << i : 0u);
    return pass;
}
__device__ __noinline__ unsigned filter_gain_pass(const FilterCtx& x, unsigned q0, int g0,
                                                  unsigned q1, int g1) {
    const int w = filter_width(x.n_D, g0);
    if (w == filter_width(x.n_D, g1)) {
        if (w == 8) return filter_gain_pass<8>(x, q0, g0, q1, g1);
        if (w == 4) return filter_gain_pass<4>(x, q0, g0, q1, g1);
        if (w == 2) return filter_gain_pass<2>(x, q0, g0, q1, g1);
        return filter_gain_pass<1>(x, q0, g0, q1, g1);
    }
    // (the second of the pair is in the last, narrower group)
    const int w1 = filter_width(x.n_D, g1);
    const unsigned p0 = filter_gain_pass<8>(x, q0, g0, q0, g0);
    const unsigned p1 = w1 == 4 ? filter_gain_pass<4>(x, q1, g1, q1, g1)
                                : (w1 == 2 ? filter_gain_pass<2>(x, q1, g1, q1, g1)
                                           : filter_gain_pass<1>(x, q1, g1, q1, g1));
    return (p0 & 0xffffu) | (p1 << 16);
}

// Bounds of four phases (Q) or one phase (S) of four durations from d0 (the
// walk from u; the odd last pair reads its own row twice).  Two epochs a
// round: a position past the end reads the empty last entry.
__device__ __noinline__ float4 filter_sums(const FilterCtx& x, unsigned long long u, int d0) {
    const FilterPeriod fp = x.fp;
    const bool quad = fp.mode == FILTER_QUAD;
    const unsigned last = (unsigned)x.f.ns - 1u, n4 = (unsigned)x.f.ns >> 2;
    const uint4* __restrict__ p0 = reinterpret_cast<const uint4*>(quad ? x.f.Q : x.f.S) +
                                   (int64_t)(d0 >> 1) * x.f.ns;
    const uint4* __restrict__ p1 = p0 + (d0 + 2 < x.n_D ? x.f.ns : 0);
    const float c = filter_slack(fp);
    float v[4], g[4], a[4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = g[i] = a[i] = b[i] = 0.f;
    if (quad) {
        auto at = [&](unsigned long long y) {
            const unsigned s = y < fp.uend ? min((unsigned)(y >> 40), last) : last;
            return (s & 3u) * n4 + (s >> 2);
        };
        auto add = [&](int i, unsigned zx, unsigned vx) {
            a[i] += __uint_as_float(zx);
            b[i] += __uint_as_float(zx << 16);
            v[i] += __uint_as_float(vx);
            g[i] += __uint_as_float(vx << 16);
        };
        for (; u < fp.uend; u += 2ull * fp.ustep) {
            const unsigned o = at(u), o2 = at(u + fp.ustep);
            const uint4 q0 = p0[o], q1 = p1[o], r0 = p0[o2], r1 = p1[o2];
            add(0, q0.x, q0.y);
            add(1, q0.z, q0.w);
            add(2, q1.x, q1.y);
            add(3, q1.z, q1.w);
            add(0, r0.x, r0.y);
            add(1, r0.z, r0.w);
            add(2, r1.x, r1.y);
            add(3, r1.z, r1.w);
        }
        const float xl = 1.f / (2.f * FILTER_BETA_B) - 1.f;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            v[i] = filter_bound(fmaxf(a[i], b[i]), v[i], g[i], FILTER_BETA_B, xl, c);
    } else {
        auto at = [&](unsigned long long y) {
            return y < fp.uend ? min((unsigned)(y >> 40), last) : last;
        };
        auto add = [&](int i, float w, unsigned zx, unsigned vx) {
            a[i] += fmaf(w, __uint_as_float(zx << 16), __uint_as_float(zx));
            v[i] += __uint_as_float(vx);
            g[i] += __uint_as_float(vx << 16);
        };
        for (; u < fp.uend; u += 2ull * fp.ustep) {
            const unsigned o = at(u), o2 = at(u + fp.ustep);
            const uint4 q0 = p0[o], q1 = p1[o], r0 = p0[o2], r1 = p1[o2];
            const float w = filter_weight(u), w2 = filter_weight(u + fp.ustep);
            add(0, w, q0.x, q0.y);
            add(1, w, q0.z, q0.w);
            add(2, w, q1.x, q1.y);
            add(3, w, q1.z, q1.w);
            add(0, w2, r0.x, r0.y);
            add(1, w2, r0.z, r0.w);
            add(2, w2, r1.x, r1.y);
            add(3, w2, r1.z, r1.w);
        }
        const float xl = 1.f / (2.f * FILTER_BETA_A) - 1.f;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            v[i] = filter_bound(a[i], v[i], g[i], FILTER_BETA_A / (1.f - FILTER_TAU), xl, c);
    }
    return make_float4(v[0], v[1], v[2], v[3]);
}

// Bounds of one phase of four durations by their gains (the only tables).
__device__ __noinline__ float4 filter_gain_sums(const FilterCtx& x, unsigned long long u, int d0) {
    const unsigned last = (unsigned)x.f.ns - 1u;
    const float* __restrict__ r = x.f.L + (int64_t)d0 * x.f.ns;
    const float ch = 1.f + filter_slack(x.fp);
    float l[4] = {0.f, 0.f, 0.f, 0.f};
    for (; u < x.fp.uend; u += x.fp.ustep) {
        const unsigned o = min((unsigned)(u >> 40), last);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (d0 + i < x.n_D) l[i] += r[(int64_t)i * x.f.ns + o];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) l[i] = l[i] > 0.f ? fmaf(l[i], ch, 0.500001f) : -INFINITY;
    return make_float4(l[0], l[1], l[2], l[3]);
}
// Q of one duration.
__device__ __forceinline__ float filter_one_quad(const FilterView& f, int d, unsigned long long u,
                                                 const FilterPeriod& fp, float c) {
    const unsigned last = (unsigned)f.ns - 1u, n4 = (unsigned)f.ns >> 2;
    const uint2* __restrict__ r = f.Q + (int64_t)(d >> 1) * f.ns * 2 + (d & 1);
    float a = 0.f, b = 0.f, v = 0.f, g = 0.f;
    for (; u < fp.uend; u += 2ull * fp.ustep) {
        const unsigned long long u2 = u + fp.ustep;
        const unsigned s = min((unsigned)(u >> 40), last);
        const unsigned s2 = u2 < fp.uend ? min((unsigned)(u2 >> 40), last) : last;
        const uint2 x = r[2u * ((s & 3u) * n4 + (s >> 2))], y = r[2u * ((s2 & 3u) * n4 + (s2 >> 2))];
        a += __uint_as_float(x.x) + __uint_as_float(y.x);
        b += __uint_as_float(x.x << 16) + __uint_as_float(y.x << 16);
        v += __uint_as_float(x.y) + __uint_as_float(y.y);
        g += __uint_as_float(x.y << 16) + __uint_as_float(y.y << 16);
    }
    return filter_bound(fmaxf(a, b), v, g, FILTER_BETA_B, 1.f / (2.f * FILTER_BETA_B) - 1.f, c);
}

// Drop the first n entries of a queue of len <= n + 32.
__device__ __forceinline__ void filter_shift_queue(uint2* q, int len, int n) {
    const int lane = threadIdx.x & 31;
    uint2 a = make_uint2(0u, 0u);
    if (n + lane < len) a = q[n + lane];
    __syncwarp();
    if (n + lane < len) q[lane] = a;
    __syncwarp();
}

// The functions below are not inlined: they run on the few groups and cells
// that pass, and inlining them into the walks' loop spills its registers.  A
// screen is a functor: screen(cnt) takes the first cnt <= 32 cells of the
// queue, one per lane.  Screen::lone: the kernel of calls that have the gains'
// tables alone (in the other kernels the walk for them costs the other walks up to
// 8 %: 420 curves of 1 700-3 700 x 7 durations x 1 000 periods, FP64, 37.7 -> 34.8 ms).
template <class Screen>
__device__ __noinline__ void filter_push_cells(FilterQueues& q, bool keep, unsigned j, unsigned d,
                                               Screen& screen) {
    const int lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    const int nc = q.nc;
    if (keep) q.cell[nc + __popc(m & ((1u << lane) - 1u))] = make_uint2(j, d);
    const int n = nc + __popc(m);
    __syncwarp();
    if (n < 32) {
        if (lane == 0) q.nc = n;
        __syncwarp();
        return;
    }
    screen(32);
    __syncwarp();
    filter_shift_queue(q.cell, n, 32);
    if (lane == 0) q.nc = n - 32;
    __syncwarp();
}
template <class Screen>
__device__ __noinline__ void filter_rest(FilterQueues& q, Screen& screen) {
    const int nc = q.nc;
    if (nc > 0) screen(nc);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) q.nc = 0;
    __syncwarp();
}
// Expand the groups at q[0 .. n) (1 << sh phases each) into cells, 32 a round.
template <class Screen>
__device__ __noinline__ void filter_expand(FilterCtx& x, FilterQueues& qs, const uint2* q, int n,
                                           int sh, Screen& screen) {
    const int lane = threadIdx.x & 31;
    for (int h = 0; h < n; h += 32 >> sh) {
        const int e = h + (lane >> sh);
        bool keep = false;
        unsigned j = 0u, d = 0u;
        if (e < n) {
            const uint2 it = q[e];
            j = (it.x << sh) + (unsigned)(lane & ((1 << sh) - 1));
            d = it.y;
            if ((int64_t)j < x.fp.n_phi) {
                // the mode's own bound first, then the other one: near K = 5
                // neither suffices alone (C2's 16-duration grid at K = 5:
                // 3.5 % of cells pass the gains alone)
                const unsigned long long u = (unsigned long long)j * x.fp.uph;
                const float c = filter_slack(x.fp);
                const bool gain = x.fp.mode == FILTER_GAIN;
                float ub = gain ? filter_one_gain(x.f, (int)d, u, x.fp, c)
                                : filter_one(x.f, (int)d, u, x.fp, c);
                keep = !(ub < filter_thr(x)) && ub != -INFINITY;
                if (!Screen::lone && keep && x.fp.K > 5.5f && x.fp.K < 14.f) {
                    ub = gain ? filter_one(x.f, (int)d, u, x.fp, c)
                              : filter_one_gain(x.f, (int)d, u, x.fp, c);
                    keep = !(ub < filter_thr(x)) && ub != -INFINITY;
                }
            }
        }
        __syncwarp();
        filter_push_cells(qs, keep, j, d, screen);
    }
}
// Queued groups of eight phases to groups of four (the quad queue), by Q: 16
// groups a round; full rounds of the quad queue go on to the cells.
template <class Screen>
__device__ __noinline__ void filter_mid(FilterCtx& x, FilterQueues& q, int n, Screen& screen) {
    const int lane = threadIdx.x & 31;
    for (int h = 0; h < n; h += 16) {
        const int e = h + (lane >> 1);
        bool keep = false;
        unsigned g = 0u, d = 0u;
        if (e < n) {
            const uint2 it = q.item[e];
            g = 2u * it.x + (unsigned)(lane & 1);
            d = it.y;
            if ((int64_t)g * 4 < x.fp.n_phi) {
                const float ub = filter_one_quad(x.f, (int)d, ((unsigned long long)g << 2) * x.fp.uph,
                                                 x.fp, filter_slack(x.fp));
                keep = !(ub < filter_thr(x)) && ub != -INFINITY;
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        const int nq = q.nq, n2 = nq + __popc(m);
        if (keep) q.quad[nq + __popc(m & ((1u << lane) - 1u))] = make_uint2(g, d);
        __syncwarp();
        const int take = n2 & ~7;
        if (take) {
            filter_expand(x, q, q.quad, take, 2, screen);
            filter_shift_queue(q.quad, n2, take);
        }
        if (lane == 0) q.nq = n2 - take;
        __syncwarp();
    }
}
// Work off the queued groups: whole rounds, or all of them at the end.
template <class Screen>
__device__ __noinline__ void filter_drain(FilterCtx& x, FilterQueues& q, bool all,
                                          Screen& screen) {
    const int lane = threadIdx.x & 31;
    const bool gain = x.fp.mode == FILTER_GAIN;
    const bool mid = !Screen::lone && gain && x.fp.K >= FILTER_K_MID + 2.f;
    const int ni = q.ni;
    const int round = mid ? 16 : (gain ? 4 : 8);
    const int n = all ? ni : ni & ~(round - 1);
    if (n > 0) {
        if (mid) filter_mid(x, q, n, screen);
        else filter_expand(x, q, q.item, n, gain ? 3 : 2, screen);
        filter_shift_queue(q.item, ni, n);
        if (lane == 0) q.ni = ni - n;
        __syncwarp();
    }
    if (all && mid) {
        filter_expand(x, q, q.quad, q.nq, 2, screen);
        if (lane == 0) q.nq = 0;
        __syncwarp();
    }
}
// The passes of one round: bit i of pass is duration d0 + i of group g.
template <class Screen>
__device__ __noinline__ void filter_take(FilterCtx& x, FilterQueues& q, unsigned pass, unsigned g,
                                         int d0, Screen& screen) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    if (x.fp.mode == FILTER_CELL) {
        for (unsigned any = __reduce_or_sync(FULL, pass); any; any &= any - 1u) {
            const int i = __ffs(any) - 1;
            filter_push_cells(q, (pass >> i) & 1u, g, (unsigned)(d0 + i), screen);
        }
        return;
    }
    const int total = __reduce_add_sync(FULL, __popc(pass));
    const int n0 = q.ni;
    __syncwarp();                          // (read by all before any lane adds)
    if (n0 + total <= FILTER_ITEMS + 32) {
        int pos = pass ? atomicAdd(&q.ni, __popc(pass)) : 0;
        for (; pass; pass &= pass - 1u)
            q.item[pos++] = make_uint2(g, (unsigned)(d0 + __ffs(pass) - 1));
        __syncwarp();
        if (q.ni >= 16) filter_drain(x, q, false, screen);
        return;
    }
    // (a first round without a threshold passes everything)
    for (unsigned any = __reduce_or_sync(FULL, pass); any; any &= any - 1u) {
        const int i = __ffs(any) - 1;
        const bool keep = (pass >> i) & 1u;
        const unsigned m = __ballot_sync(FULL, keep);
        const int ni = q.ni;
        if (keep) q.item[ni + __popc(m & ((1u << lane) - 1u))] = make_uint2(g, (unsigned)(d0 + i));
        __syncwarp();
        if (lane == 0) q.ni = ni + __popc(m);
        __syncwarp();
        filter_drain(x, q, false, screen);
    }
}
// The largest finite bound b > 0 of a warp's first round (duration d of group
// g) goes through the screen at once: its lower bound seeds the threshold.
template <class Screen>
__device__ __noinline__ void filter_seed(FilterCtx& x, FilterQueues& q, float b, unsigned g,
                                         int d, Screen& screen) {
    const unsigned FULL = 0xffffffffu;
    const unsigned k = b > 0.f && b < INFINITY ? __float_as_uint(b) : 0u;
    const unsigned top = __reduce_max_sync(FULL, k);
    if (!top) return;
    const int src = __ffs(__ballot_sync(FULL, k == top)) - 1;
    const unsigned g1 = __shfl_sync(FULL, g, src);
    const int d1 = __shfl_sync(FULL, d, src);
    const int lane = threadIdx.x & 31;
    const int sh = filter_shift(x.fp.mode);
    const unsigned j = (g1 << sh) + (unsigned)lane;
    filter_push_cells(q, lane < (1 << sh) && (int64_t)j < x.fp.n_phi, j, (unsigned)d1, screen);
    filter_rest(q, screen);
}

// The groups of one mode, in the order the warps take them.
struct FilterGroups {
    unsigned nq, n_it, stride;
    int W;                 // durations of a group
    __device__ __forceinline__ void advance(unsigned& q, int& g) const {
        q += stride;
        while (q >= nq) {
            q -= nq;
            ++g;
        }
    }
};
// Seed from a warp's first round: the largest bound of its lanes' first groups.
template <class Screen>
__device__ __noinline__ void filter_first(FilterCtx& x, FilterQueues& q, bool act, unsigned qi,
                                          int gi, Screen& screen) {
    float b = 0.f;
    int bd = 0;
    const int n_D = x.n_D;
    if (x.fp.mode == FILTER_GAIN) {
        const int d0 = gi * 8;
        if (act) {
            FilterGains s;
            const int w = filter_width(n_D, gi);
            if (w == 8) filter_gains<8>(x, qi, gi, qi, gi, s);
            else if (w == 4) filter_gains<4>(x, qi, gi, qi, gi, s);
            else if (w == 2) filter_gains<2>(x, qi, gi, qi, gi, s);
            else filter_gains<1>(x, qi, gi, qi, gi, s);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (s.a[i] > b && s.a[i] < INFINITY) {
                    b = s.a[i];
                    bd = i;
                }
        }
        bd += d0;
    } else {
        const int d0 = gi * 4;
        if (act) {
            const float4 u = filter_sums(x, ((unsigned long long)qi << filter_shift(x.fp.mode)) *
                                                x.fp.uph, d0);
            const float ub[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (d0 + i < n_D && ub[i] > b && ub[i] < INFINITY) {
                    b = ub[i];
                    bd = i;
                }
        }
        bd += d0;
    }
    filter_seed(x, q, b, qi, bd, screen);
}

// The cells of a period by their gains, four durations a lane (FILTER_LONE).
template <class Screen>
__device__ __noinline__ void filter_lone(FilterCtx& x, int wid, int nw, FilterQueues& q,
                                         Screen& screen) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned n_phi = (unsigned)x.fp.n_phi;
    const unsigned n_it = n_phi * (unsigned)((x.n_D + 3) / 4);
    bool first = true;
    for (unsigned base = (unsigned)wid * 32u; base < n_it; base += (unsigned)nw * 32u) {
        const unsigned i = base + (unsigned)lane;
        const int gi = (int)(i / n_phi), d0 = 4 * gi;
        const unsigned j = i - (unsigned)gi * n_phi;
        float ub[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        if (i < n_it) {
            const float4 u = filter_gain_sums(x, (unsigned long long)j * x.fp.uph, d0);
            ub[0] = u.x;
            ub[1] = u.y;
            ub[2] = u.z;
            ub[3] = u.w;
        }
        if (first) {
            float b = 0.f;
            int bd = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (d0 + k < x.n_D && ub[k] > b && ub[k] < INFINITY) {
                    b = ub[k];
                    bd = k;
                }
            filter_seed(x, q, b, j, d0 + bd, screen);
            first = false;
        }
        const float t = filter_thr(x);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool keep = d0 + k < x.n_D && !(ub[k] < t) && ub[k] != -INFINITY;
            if (__any_sync(FULL, keep)) filter_push_cells(q, keep, j, (unsigned)(d0 + k), screen);
        }
    }
    filter_rest(q, screen);
}

// Runs the filters over every cell of a period.  The item's warps (wid of
// nw) share the work.  Cells below the threshold are dropped, the others go
// through the screen.
template <class Screen>
__device__ __forceinline__ void filter_cells(FilterCtx& x, int wid, int nw, FilterQueues& q,
                                             Screen& screen) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int n_D = x.n_D, mode = x.fp.mode;
    if constexpr (Screen::lone) {
        if (mode == FILTER_LONE) {
            filter_lone(x, wid, nw, q, screen);
            return;
        }
    }
    const int sh = filter_shift(mode);
    FilterGroups g;
    g.W = mode == FILTER_GAIN ? 8 : 4;
    g.nq = (unsigned)((x.fp.n_phi + (1 << sh) - 1) >> sh);
    g.n_it = g.nq * (unsigned)((n_D + g.W - 1) / g.W);
    g.stride = (unsigned)nw * 32u;
    unsigned i = (unsigned)(wid * 32 + lane);            // this lane's group
    int gi = (int)(i / g.nq);
    unsigned qi = i - (unsigned)gi * g.nq;
    if ((unsigned)wid * 32u < g.n_it) filter_first(x, q, i < g.n_it, qi, gi, screen);
    auto mask = [&](unsigned pass, int d0) {             // durations past the last
        return d0 + g.W > n_D ? (d0 < n_D ? pass & ((1u << (n_D - d0)) - 1u) : 0u) : pass;
    };
    if (mode == FILTER_GAIN) {
        for (unsigned base = (unsigned)wid * 32u; base < g.n_it;
             base += 2u * g.stride, i += 2u * g.stride) {
            unsigned q1 = qi;
            int g1 = gi;
            g.advance(q1, g1);
            const bool in0 = i < g.n_it, in1 = in0 && i + g.stride < g.n_it;
            unsigned pass = 0u;
            if (in0) pass = filter_gain_pass(x, qi, gi, in1 ? q1 : qi, in1 ? g1 : gi);
            const int d0 = gi * g.W, d1 = g1 * g.W;
            const unsigned p0 = mask(pass & 0xffffu, d0), p1 = in1 ? mask(pass >> 16, d1) : 0u;
            if (__any_sync(FULL, (p0 | p1) != 0u)) {
                filter_take(x, q, p0, qi, d0, screen);
                filter_take(x, q, p1, q1, d1, screen);
            }
            qi = q1;
            gi = g1;
            g.advance(qi, gi);
        }
    } else {
        for (unsigned base = (unsigned)wid * 32u; base < g.n_it;
             base += g.stride, i += g.stride) {
            const int d0 = gi * 4;
            unsigned pass = 0u;
            if (i < g.n_it) {
                const float4 u = filter_sums(x, ((unsigned long long)qi << sh) * x.fp.uph, d0);
                const float t = filter_thr(x);
                pass = (!(u.x < t) && u.x != -INFINITY ? 1u : 0u) |
                       (!(u.y < t) && u.y != -INFINITY ? 2u : 0u) |
                       (!(u.z < t) && u.z != -INFINITY ? 4u : 0u) |
                       (!(u.w < t) && u.w != -INFINITY ? 8u : 0u);
                pass = mask(pass, d0);
            }
            if (__any_sync(FULL, pass != 0u)) filter_take(x, q, pass, qi, d0, screen);
            g.advance(qi, gi);
        }
    }
    if (mode != FILTER_CELL) filter_drain(x, q, true, screen);
    filter_rest(q, screen);
}

}  // namespace nu
