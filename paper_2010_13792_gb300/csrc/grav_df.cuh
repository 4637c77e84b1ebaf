// FP64-accurate pair sums in two-part FP32 arithmetic ("double-float").
//
// GB300 runs FP64 at 1/64 of its FP32 rate (2 FMA per clock and SM), and the
// FP64 force kernel needs 39 FP64 instructions a pair: 2500 FP32 lane slots.
// The same pair carried as unevaluated sums of two FP32 numbers (about 48 bits)
// takes some 320 FP32 operations, two sources to a packed FP32x2 instruction
// (ncu: 203 warp instructions a pair with everything around them).
//
// Pieces:
//   * Tiles hold the sources' offsets from the tile centre in units of a power
//     of two L, velocities in units V and masses in units of the largest mass
//     M, so the FP32 range does not limit the caller's units and the rounding
//     of a mass that all sources share does not bias the sums (it would be the
//     same 2^-49 for each): x = sh + sl, each rounded to nearest.
//   * Separations: Knuth's TwoSum of the high parts plus the difference of the
//     low parts, renormalised.
//   * r^-3 and r^-5 from y, the SFU's rsqrt after one FP32 Newton step: with
//     t = 1 - r^2 y^2 formed from both parts, r^-3 = y^3 (1 + 3/2 t + 15/8 t^2),
//     r^-2 = y^2 (1 + t + t^2) (the binomial series; |t| <= 2^-22, so the next
//     terms are below 2^-64).
//   * Sums: a product's high part p is split at the unit of a constant C =
//     1.5 * 2^k that exceeds every |p|: p + C holds p rounded to a multiple of
//     ulp(C) in its low mantissa bits, which are added up exactly as integers
//     (one three-input integer add for two sources); the rest, exact, is cut
//     a second time at the unit of a smaller constant, and what then remains
//     joins the product's low part in an FP32 sum.  Nothing but that last sum
//     is rounded, and it is 2^20 and more below the total even where the window
//     is a thousand times wider than the sum.
// A pair comes out good to about 8e-15 (rms, its force; FP64 3e-16), and the
// terms of a tile average that.  What would not average is summed in FP64: the
// pairs closest to a target (listed), sources that carry a tile and tiles whose
// terms cancel (kDfAverage).
#pragma once

#include "grav_common.cuh"

namespace grav {

// Words of a packed tile of S sources: an 8-word header, the boxes of its
// sub-blocks of 32 sources (lo, hi in units of L, rounded outward), a word per
// sub-block that marks its heavy sources (a multiple of 4 words so far), S/2
// records of 28 floats (two sources side by side: xh yh zh xl yl zl, the same
// of the velocity, mh ml; heavy sources and padding with mass and velocity 0).
constexpr int kDfSub = 32;
constexpr int kDfHeader = 8;
template <int S>
constexpr int df_heavies() { return kDfHeader + 6 * (S / kDfSub); }
template <int S>
constexpr int df_records() { return (df_heavies<S>() + S / kDfSub + 3) / 4 * 4; }
template <int S>
constexpr int df_words() { return df_records<S>() + 14 * S; }
template <int S>
constexpr uint32_t df_bytes() { return 4u * df_words<S>(); }
// stride of the tiles in the workspace
constexpr int64_t kDfBytesPerSource = 58;
template <int S>
constexpr int64_t df_stride() { return kDfBytesPerSource * S; }
static_assert(df_bytes<64>() <= df_stride<64>() && df_bytes<128>() <= df_stride<128>() &&
              df_bytes<256>() <= df_stride<256>() && df_stride<64>() % 16 == 0, "DF tile stride");

struct DfHead {
    double munit;      // M: the largest |m| but for the heavy ones (1 if all are 0)
    float ext[3];      // half extents / L, rounded up
    int16_t el, ev;    // units: L = 2^el >= half extent, V = 2^ev > |v'|
    int16_t ok;        // 0: the tile is summed in FP64 (out of range, or its terms do not average)
    int16_t count;     // sources in the tile
    int32_t pad;
};
static_assert(sizeof(DfHead) == 4 * kDfHeader, "DfHead layout");

// A power of two above |x| of the largest high word hi (of |x|).
__device__ __forceinline__ int exponent_above(uint32_t hi) { return (int)(hi >> 20) - 1022; }

__device__ __forceinline__ double pow2d(int e)   // -1022 <= e <= 1023
{
    return __hiloint2double((e + 1023) << 20, 0);
}

__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
// a - b, rounded once
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, dup2(-1.0f), a); }

// Sources that carry a tile.  A two-part pair term is good to some 8e-15 of
// itself, thirty times FP64's rounding; the sums are as good as FP64's where many
// like terms average it away, and not where a few terms carry a sum, nor where the
// windows, which the largest attribute sets, belong to a source that the target
// does not sum (itself): terms below 2^-42 of the window are plain FP32.  So
// with w the masses (and the |v'|, or the a_bar) of the tile:
//   * the tile averages if sum w^2 <= (sum w)^2 / K, the largest w left out of
//     the right side (a target does not sum itself), K = 64: a spread of
//     masses, up to 64 equal ones (fewer in a ragged last tile);
//   * otherwise the sources above sum w / (2 K + 2) are heavy, at most 2 K + 3 of
//     them: they are summed in FP64, and the rest averages, since its sum of
//     squares is at most its largest times its sum, sum w^2 <= 2 (sum w)^2 / (2 K + 2);
//   * a tile whose w cancel (|sum w| < sum |w| / 2, an a_bar of random signs) is
//     summed in FP64 altogether, and so are systems of up to 128 elements.
// Measured (rms error of the acceleration; FP64 pairs / two parts alone / with
// this rule): 10000-element Plummer sphere, masses from 0.1 to 100 with their
// number falling as m^-2.35 1.7e-16 / 9.9e-16 / 2.4e-16, over 14 decades 2.2e-16 /
// 1.1e-15 / 1.4e-16; one mass of 1 among 299 of 1e-12, at it, 3.8e-16 / 3.1e-9 /
// 6.8e-16; the adjoint's largest error for a random a_bar 3e-15 / 6e-14 / 3e-15.
// 16384 elements: 4.4 ms, with that mass function 5.1 ms.
// For an a_bar K = 16 (2e-15 of the tile's sum): in the middle of a smooth field it
// points to all sides, and |sum| is a third of the sum of its norms; such a tile is one
// of many.  A smooth loss, forward and adjoint, K = 64 / 16: sphere of 1771 908 / 841 us, cloud of
// 3000 1434 / 1288 us, with the same errors; random signs still go to FP64.
constexpr int kDfAverage = 64, kDfAverageAdj = 16;
constexpr int kDfFewest = 128;

// (the larger side of the rule: heavier than this)
__device__ __forceinline__ float df_heavy_line(float net, float gross, float squares, float K, bool &ok)
{
    if (squares * K <= net * net) return __int_as_float(0x7f800000);
    if (gross > 2.0f * net) ok = false;
    return net / (2.0f * K + 2.0f);
}

// Packs one tile (one CTA of S threads, thread j its source): `x` the FP64
// offset from the tile centre, `v` the velocity relative to the tile's
// velocity centre (ADJ: the adjoint's a_bar), m the mass; `half` the tile's half
// extents; `alone`: the system has no other tile; all_fp64: the caller wants every
// tile summed in FP64.  Padding sources (!ok) copy the
// place of their sub-block's first source with zero mass.  A warp is a sub-block.
template <int S, bool ADJ>
__device__ __forceinline__ void df_pack(void *tile, int j, bool ok, int count, bool alone, bool all_fp64,
                                        const double x[3], const double v[3], double m, const double half[3],
                                        double cmax)
{
    constexpr int W = S / 32;
    __shared__ uint32_t wtop[2][W], wlight[3][W];
    __shared__ int wat[2][W];
    __shared__ float wsum[8][W];
    const int lane = j & 31, wid = j >> 5;
    // the largest mass and velocity (by the high words), and who has them
    uint32_t hv = 0, hm = 0;
    if (ok) {
#pragma unroll
        for (int c = 0; c < 3; ++c) hv = max(hv, (uint32_t)__double2hiint(v[c]) & 0x7fffffffu);
        hm = (uint32_t)__double2hiint(m) & 0x7fffffffu;
    }
    {
        const uint32_t tm = __reduce_max_sync(0xffffffffu, hm), tv = __reduce_max_sync(0xffffffffu, hv);
        const int am = __ffs(__ballot_sync(0xffffffffu, ok && hm == tm)) - 1;
        const int av = __ffs(__ballot_sync(0xffffffffu, ok && hv == tv)) - 1;
        if (lane == 0) {
            wtop[0][wid] = tm;
            wtop[1][wid] = tv;
            wat[0][wid] = am;
            wat[1][wid] = av;
        }
    }
    __syncthreads();
    uint32_t top[2] = {0u, 0u};
    int at[2] = {-1, -1};
#pragma unroll
    for (int w = 0; w < W; ++w)
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if (wat[c][w] >= 0 && (at[c] < 0 || wtop[c][w] > top[c])) {
                top[c] = wtop[c][w];
                at[c] = 32 * w + wat[c][w];
            }
    uint32_t hx = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) hx = max(hx, (uint32_t)__double2hiint(half[c]) & 0x7fffffffu);
    // L no smaller than 2^-10 of the centre's distance from the origin: targets
    // of a tile of coincident elements stay in range
    const uint32_t hc = (uint32_t)__double2hiint(cmax) & 0x7fffffffu;
    DfHead h;
    int el = max(exponent_above(hx), exponent_above(hc) - 10);
    if (hx == 0 && hc == 0) el = 0;
    const int em = top[0] == 0 ? 0 : exponent_above(top[0]), ev = top[1] == 0 ? 0 : exponent_above(top[1]);
    bool good = hx < 0x7ff00000u && top[0] < 0x7ff00000u && top[1] < 0x7ff00000u && abs(el) <= 150 &&
                abs(em) <= 150 && abs(ev) <= 150 && !(alone && count <= kDfFewest) && !all_fp64;
    el = max(-150, min(150, el));
    h.el = (int16_t)el;
    // heavy sources
    float w = 0.0f, u[3] = {0.0f, 0.0f, 0.0f};
    if (ok && good) {
        const double im = pow2d(-em), iv = pow2d(-ev);
        w = __double2float_rn(__dmul_rn(m, im));
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] = __double2float_rn(__dmul_rn(v[c], iv));
    }
    const float uu = fmaf(u[0], u[0], fmaf(u[1], u[1], u[2] * u[2])), un = sqrtf(uu);
    const bool not_m = j != at[0], not_v = j != at[1];
    float sum[8] = {not_m ? w : 0.0f,    not_m ? fabsf(w) : 0.0f, w * w,
                    not_v ? u[0] : 0.0f, not_v ? u[1] : 0.0f,     not_v ? u[2] : 0.0f,
                    not_v ? un : 0.0f,   uu};
    constexpr int kFirst = ADJ ? 3 : 0;
#pragma unroll
    for (int q = kFirst; q < 8; ++q) {
        if (!ADJ && q >= 3 && q < 6) continue;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum[q] += __shfl_xor_sync(0xffffffffu, sum[q], o);
        if (lane == 0) wsum[q][wid] = sum[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = kFirst; q < 8; ++q) {
        if (!ADJ && q >= 3 && q < 6) continue;
        sum[q] = 0.0f;
#pragma unroll
        for (int k = 0; k < W; ++k) sum[q] += wsum[q][k];
    }
    const float K = fminf((float)(ADJ ? kDfAverageAdj : kDfAverage), 0.5f * (float)count);
    const float net_v = ADJ ? sqrtf(fmaf(sum[3], sum[3], fmaf(sum[4], sum[4], sum[5] * sum[5]))) : sum[6];
    bool heavy = un > df_heavy_line(net_v, sum[6], sum[7], K, good);
    if (!ADJ) heavy = fabsf(w) > df_heavy_line(fabsf(sum[0]), sum[1], sum[2], K, good) || heavy;
    // the units are those of the others
    const uint32_t marks = __ballot_sync(0xffffffffu, heavy);
    {
        uint32_t lm = (uint32_t)__double2loint(m);
        if (!ok || heavy) hv = hm = lm = 0;
        const uint32_t tv = __reduce_max_sync(0xffffffffu, hv), tm = __reduce_max_sync(0xffffffffu, hm);
        lm = __reduce_max_sync(0xffffffffu, hm == tm ? lm : 0u);
        if (lane == 0) {
            wlight[0][wid] = tv;
            wlight[1][wid] = tm;
            wlight[2][wid] = lm;
        }
    }
    __syncthreads();
    hv = hm = 0;
    uint32_t lm = 0;
#pragma unroll
    for (int k = 0; k < W; ++k) {
        hv = max(hv, wlight[0][k]);
        const uint32_t h2 = wlight[1][k], l2 = wlight[2][k];
        lm = h2 > hm ? l2 : h2 == hm ? max(lm, l2) : lm;
        hm = max(hm, h2);
    }
    // (the sums above are FP32: they say nothing of what lies 2^96 below)
    good = good && (hm == 0 || exponent_above(hm) >= em - 96) && (hv == 0 || exponent_above(hv) >= ev - 96);
    h.ok = good;
    h.ev = (int16_t)(good && hv != 0 ? exponent_above(hv) : 0);
    h.munit = good && hm != 0 ? __hiloint2double((int)hm, (int)lm) : 1.0;
    h.count = (int16_t)count;
    h.pad = 0;
    const double il = pow2d(-el);
#pragma unroll
    for (int c = 0; c < 3; ++c) h.ext[c] = __double2float_ru(__dmul_rn(half[c], il));
    float *out = static_cast<float *>(tile);
    if (j == 0) *reinterpret_cast<DfHead *>(out) = h;
    const double iv = pow2d(-h.ev);
    float *rec = out + df_records<S>() + 28 * (j >> 1) + (j & 1);
    float *box = out + kDfHeader + 6 * wid;
    if (lane == 0) reinterpret_cast<uint32_t *>(out)[df_heavies<S>() + wid] = good ? marks : 0u;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double s = __shfl_sync(0xffffffffu, __dmul_rn(x[c], il), ok ? lane : 0);
        const float sh = __double2float_rn(s);
        rec[2 * c] = sh;
        rec[6 + 2 * c] = __double2float_rn(__dsub_rn(s, (double)sh));
        float lo = __double2float_rd(s), hi = __double2float_ru(s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if (lane == 0) {
            box[c] = lo;
            box[3 + c] = hi;
        }
        const double vu = ok && !heavy ? __dmul_rn(v[c], iv) : 0.0;
        const float vh = __double2float_rn(vu);
        rec[12 + 2 * c] = vh;
        rec[18 + 2 * c] = __double2float_rn(__dsub_rn(vu, (double)vh));
    }
    const double mw = ok && !heavy ? __ddiv_rn(m, h.munit) : 0.0;
    const float mh = __double2float_rn(mw);
    rec[24] = mh;
    rec[26] = __double2float_rn(__dsub_rn(mw, (double)mh));
}

// A target against one tile: offset from the tile centre in units of L, in
// three parts (a pair's separation needs two; the third keeps the offset's own
// rounding, which all pairs of the tile share, out of the sums).
struct DfTarget {
    float h[3], l[3], l2[3];
};

__device__ __forceinline__ void df_split(const double x[3], DfTarget &t)
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        t.h[c] = __double2float_rn(x[c]);
        const double r1 = __dsub_rn(x[c], (double)t.h[c]);
        t.l[c] = __double2float_rn(r1);
        t.l2[c] = __double2float_rn(__dsub_rn(r1, (double)t.l[c]));
    }
}

// C = 1.5 * 2^k with 2^(k-1) > b (b > 0, normal).
__device__ __forceinline__ float df_window(float b)
{
    return __uint_as_float((__float_as_uint(b) & 0x7f800000u) + (2u << 23) + 0x400000u);
}

// One two-part sum of a target over a tile: i1 counts units ulp(C), i2 units
// ulp(C2), lo the rest (its two lanes the even and the odd sources).
struct DfSum {
    uint32_t i1, i2;
    float2 lo;
};

// Second window of a sum: 2^4 units of C, so |rest| may reach 8 units.
__device__ __forceinline__ float df_second(float C) { return __uint_as_float(__float_as_uint(C) - (19u << 23)); }

// Moves the part of `lo` above ulp(C2) into the second integer sum.
__device__ __forceinline__ void df_carry(DfSum &s, float2 C2)
{
    const float2 t = __fadd2_rn(s.lo, C2);
    s.i2 += __float_as_uint(t.x) + __float_as_uint(t.y);
    s.lo = __fadd2_rn(s.lo, sub2(C2, t));
}

// sum += (fh + fl) (dh + dl) for two sources; df_carry follows every
// kDfCarry records.
constexpr int kDfCarry = 8;

__device__ __forceinline__ void df_add_product(DfSum &s, float2 C, float2 C2, float2 fh, float2 fl,
                                               float2 dh, float2 dl)
{
    const float2 p = __fmul2_rn(fh, dh);
    float2 w = __ffma2_rn(fh, dh, neg2(p));
    w = __ffma2_rn(fh, dl, w);
    w = __ffma2_rn(fl, dh, w);
    const float2 t = __fadd2_rn(p, C);
    s.i1 += __float_as_uint(t.x) + __float_as_uint(t.y);
    const float2 r = __fadd2_rn(p, sub2(C, t));
    const float2 u = __fadd2_rn(r, C2);
    s.i2 += __float_as_uint(u.x) + __float_as_uint(u.y);
    s.lo = __fadd2_rn(s.lo, __fadd2_rn(__fadd2_rn(r, sub2(C2, u)), w));
}

// The sum as FP64 in the caller's units (`unit` of the tile's), after n1
// additions to i1 and n2 to i2.
__device__ __forceinline__ double df_value(const DfSum &s, float C, uint32_t n1, uint32_t n2, double unit)
{
    const int a = (int)(s.i1 - n1 * __float_as_uint(C));
    const int b = (int)(s.i2 - n2 * __float_as_uint(df_second(C)));
    const long long n = ((long long)a << 19) + b;
    const int e2 = (int)(__float_as_uint(C) >> 23) - 127 - 42;          // ulp(C2) = 2^e2
    // (`unit` is normal and far from the ends: its exponent can be moved)
    const double scale = __hiloint2double(__double2hiint(unit) + (e2 << 20), __double2loint(unit));
    return __fma_rn((double)n, scale, __dmul_rn((double)__fadd_rn(s.lo.x, s.lo.y), unit));
}

// (ah + al) (bh + bl), high and low parts not renormalised.
__device__ __forceinline__ void df_mul(float2 ah, float2 al, float2 bh, float2 bl, float2 &ph, float2 &pl)
{
    ph = __fmul2_rn(ah, bh);
    pl = __ffma2_rn(ah, bh, neg2(ph));
    pl = __ffma2_rn(ah, bl, pl);
    pl = __ffma2_rn(al, bh, pl);
}

__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = __fadd2_rn(a, b);
    const float2 z = sub2(s, a);
    e = __fadd2_rn(sub2(a, sub2(s, z)), sub2(b, z));
}

// h + l renormalised (|h| >= |l|): |l| at most half a unit of h.
__device__ __forceinline__ void df_norm(float2 &h, float2 &l)
{
    const float2 s = __fadd2_rn(h, l);
    l = sub2(l, sub2(s, h));
    h = s;
}

// Separation component: source (sh, sl) minus target (n*: its parts negated).
__device__ __forceinline__ void df_diff(float2 sh, float2 sl, float nh, float nl, float n2, float2 &d,
                                        float2 &e)
{
    two_sum2(sh, dup2(nh), d, e);
    e = __fadd2_rn(e, __fadd2_rn(sl, dup2(nl)));
    df_norm(d, e);
    e = __fadd2_rn(e, dup2(n2));
}

// Sum of three products (high parts TwoSum'd, not renormalised).
__device__ __forceinline__ void df_dot3(const float2 ah[3], const float2 al[3], const float2 bh[3],
                                        const float2 bl[3], float2 &ph, float2 &pl)
{
    float2 h[3], l[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) df_mul(ah[c], al[c], bh[c], bl[c], h[c], l[c]);
    float2 s, e1, e2;
    two_sum2(h[0], h[1], s, e1);
    two_sum2(s, h[2], ph, e2);
    pl = __fadd2_rn(__fadd2_rn(__fadd2_rn(l[0], l[1]), l[2]), __fadd2_rn(e1, e2));
}

// r^2, renormalised, without the squares of the low parts: those lie below
// the last place of the result.  Being of one sign they would not average over
// the pairs; their sum (sq) goes into the series instead (DfInv::s).
__device__ __forceinline__ void df_square3(const float2 d[3], const float2 e[3], float2 &ph, float2 &pl,
                                           float2 &sq)
{
    float2 h[3], l[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        h[c] = __fmul2_rn(d[c], d[c]);
        l[c] = __ffma2_rn(__fadd2_rn(d[c], d[c]), e[c], __ffma2_rn(d[c], d[c], neg2(h[c])));
    }
    sq = __ffma2_rn(e[0], e[0], __ffma2_rn(e[1], e[1], __fmul2_rn(e[2], e[2])));
    float2 s, e1, e2;
    two_sum2(h[0], h[1], s, e1);
    two_sum2(s, h[2], ph, e2);
    pl = __fadd2_rn(__fadd2_rn(__fadd2_rn(l[0], l[1]), l[2]), __fadd2_rn(e1, e2));
    df_norm(ph, pl);
}

// y = r^-1, t = 1 - r^2 y^2, y^2 as two parts, and s = -sq y^2, the part of t
// below its last place (it is added to a product inside an fma, whose own
// low bits keep it from being rounded away).
struct DfInv {
    float2 y, t, y2h, y2l, s;
};

__device__ __forceinline__ DfInv df_inverse(float2 r2h, float2 r2l, float2 sq)
{
    DfInv v;
    const float2 n = neg2(r2h);
    const float2 y0 = make_float2(rsqrt_sfu(r2h.x), rsqrt_sfu(r2h.y));
    v.y = __ffma2_rn(__fmul2_rn(dup2(0.5f), y0), __ffma2_rn(__fmul2_rn(n, y0), y0, dup2(1.0f)), y0);
    v.y2h = __fmul2_rn(v.y, v.y);
    v.y2l = __ffma2_rn(v.y, v.y, neg2(v.y2h));
    float2 t = __ffma2_rn(n, v.y2h, dup2(1.0f));
    t = __ffma2_rn(n, v.y2l, t);
    v.t = __ffma2_rn(neg2(r2l), v.y2h, t);
    v.s = __fmul2_rn(neg2(sq), v.y2h);
    return v;
}

// r^-3 (two parts).
__device__ __forceinline__ void df_inv3(const DfInv &v, float2 &h, float2 &l)
{
    const float2 c = __ffma2_rn(v.t, __ffma2_rn(dup2(1.875f), v.t, dup2(1.5f)), __fmul2_rn(dup2(1.5f), v.s));
    h = __fmul2_rn(v.y2h, v.y);
    l = __ffma2_rn(v.y2h, v.y, neg2(h));
    l = __ffma2_rn(v.y2l, v.y, l);
    l = __ffma2_rn(h, c, l);
    df_norm(h, l);
}

// Times r^-2.
__device__ __forceinline__ void df_times_inv2(const DfInv &v, float2 fh, float2 fl, float2 &gh, float2 &gl)
{
    float2 h = v.y2h, l = __ffma2_rn(v.y2h, __ffma2_rn(v.t, v.t, v.t), v.y2l);
    df_norm(h, l);
    df_mul(fh, fl, h, l, gh, gl);
}

// Windows of one target against one tile (units of L, V, M): every term of an
// accumulated sum stays below half its window's power of two.
struct DfWindows {
    float a, t, j, p;
};

// rmin2 <= r^2 of every pair that is summed.
__device__ __forceinline__ DfWindows df_windows(float rmin2)
{
    DfWindows w;
    const float i1 = rsqrt_sfu(rmin2) * (1.0f + 0x1p-18f);
    const float i2 = i1 * i1;
    w.a = df_window(i2);                 // m f d     <= r^-2
    w.t = df_window(i2 * i1);            // m g d d   <= r^-3
    w.j = df_window(1.8f * (i2 * i1));   // m f v <= r^-3, m g (d.v) d <= sqrt(3) r^-3 (|v_c| <= 1)
    w.p = df_window(i1);                 // m phi     <= r^-1
    return w;
}

// Where a tile's sub-blocks lie for the targets of a warp (one per lane).
constexpr float kDfRange = 32768.0f;   // targets beyond this many L from a tile: FP64
// Pairs closer than this share of the sub-block's diagonal (2.3 spacings of
// its sources) are listed for FP64, and so are softened pairs.
constexpr float kDfNear = 0.42f;
constexpr int kDfList = 64;            // room for two sub-blocks per target
// Least r^2 / L^2 in two parts: from there m r^-5 stays below 2^110 in FP32.  L is
// at least 2^-10 of the tile's distance from the origin, so a tile a billion
// times smaller than that distance has pairs below it (r^-5 ran over in the
// jerk and the tidal tensor); it is right for targets farther away.
constexpr float kDfLeast2 = 0x1p-44f;
// Elements need not come in spatial order: a sub-block of scattered sources is as
// long as the system, most of its pairs are close, and listing them one by one
// costs more than summing the sub-block in FP64.  So the forward counts them first
// (FP32, 2% of a sub-block's two-part sums), and above this share the sub-block goes
// to FP64.  Plummer spheres in random order, FP64 pairs / listed / by this rule:
// 16384 elements 19.7 / 25.7 / 20.6 ms, 65536 312 / 407 / 326 ms; in Morton order 65536
// 54.8 ms either way.  Shares from 0.2 to 0.5 do alike in random order, from 0.65 a
// uniform sphere loses it; in Morton order 0.35 lists more of the nearest sub-blocks
// than 0.25 (cloud of 6794 1.48 -> 1.41 ms).
// The adjoint lists: 12289 7.64 ms against 7.74 in FP64 tiles.
constexpr float kDfLoose = 0.35f;

struct DfClass {
    uint32_t direct;   // sub-blocks summed in FP64 (softening wider than half their diagonal, kDfLeast2)
    uint32_t loose;    // of these, those with too many pairs to list
    uint32_t close;    // sub-blocks with listed pairs
    float rmin2;       // least r^2 of the pairs left to this lane's target
    float floor2;      // least listing radius (squared)
};

// The heavy sources of sub-block q.
template <int S>
__device__ __forceinline__ uint32_t df_heavy(const float *tile, int q)
{
    return reinterpret_cast<const uint32_t *>(tile)[df_heavies<S>() + q];
}

// The sources of a sub-block of `real` that go to FP64 one by one.
template <int S>
__device__ __forceinline__ uint32_t df_fp64_sources(const float *tile, uint32_t direct, int q, int real)
{
    return (direct >> q) & 1u ? 0xffffffffu >> (kDfSub - real) : df_heavy<S>(tile, q);
}

// The marked sources of a sub-block spread over a warp, the k-th of them on lane
// k: this lane's source (the last one again past the end), and which of them is
// the element `self` of the sub-block, this lane's target (-1: none).
struct DfMarked {
    int own, count, self;
    __device__ __forceinline__ DfMarked(uint32_t marks, int64_t target)
    {
        count = __popc(marks);
        self = target >= 0 && target < kDfSub && (marks >> (int)target & 1u)
                   ? __popc(marks & ((1u << (int)target) - 1u)) : -1;
        own = min((int)(threadIdx.x & 31u), count - 1);
        if (marks & (marks + 1u)) own = (int)__fns(marks, 0, own + 1);   // (not the first `count` of them)
    }
};

template <int S>
__device__ __forceinline__ bool df_any_fp64(const float *tile, uint32_t direct, int n_sub)
{
    uint32_t any = direct;
    for (int q = 0; q < n_sub; ++q) any |= df_heavy<S>(tile, q);
    return any != 0;
}

// The softening of the FP64 pair terms, formed once per tile (the division alone is
// some 20 FP64 instructions, most of a pair).
struct DfSoftening {
    double h2, hinv, hinv3, hinv5;
    __device__ __forceinline__ explicit DfSoftening(double h)
    {
        h2 = h * h;
        hinv = 1.0 / h;
        hinv3 = hinv * hinv * hinv;
        hinv5 = hinv3 * hinv * hinv;
    }
};

__device__ __forceinline__ float df_diagonal2(const float *box)
{
    float d = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) d = fmaf(box[3 + c] - box[c], box[3 + c] - box[c], d);
    return d;
}

__device__ __forceinline__ float df_radius2(const DfClass &k, float diag2)
{
    return fmaxf(k.floor2, kDfNear * kDfNear * diag2);
}

// How many of the `real` sources of sub-block q lie within sqrt(thr2) of this
// lane's target (FP32, high parts).
template <int S>
__device__ __forceinline__ int df_count_close(const float *tile, int q, int real, const DfTarget &tg, float thr2)
{
    const float4 *P = reinterpret_cast<const float4 *>(tile + df_records<S>()) + 7 * (kDfSub / 2) * q;
    int n = 0;
    for (int k = 0; k < (real + 1) / 2; ++k) {
        const float4 a = P[7 * k];                                           // x x y y
        const float2 b = *reinterpret_cast<const float2 *>(P + 7 * k + 1);   // z z
        const float2 dx = __fadd2_rn(make_float2(a.x, a.y), dup2(-tg.h[0]));
        const float2 dy = __fadd2_rn(make_float2(a.z, a.w), dup2(-tg.h[1]));
        const float2 dz = __fadd2_rn(b, dup2(-tg.h[2]));
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        n += (r2.x < thr2) + (r2.y < thr2);
    }
    return n;
}

// h: the support in the caller's units, il = 1 / L.  LOOSE: sub-blocks with more
// than kDfLoose of their pairs to list are summed in FP64.
template <int S, bool LOOSE>
__device__ __forceinline__ DfClass df_classify(const float *tile, const DfHead &head, const DfTarget &tg,
                                               bool live, double h, double il)
{
    DfClass k;
    float at = 0.0f, ext2 = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        at = fmaxf(at, fabsf(tg.h[c]));
        ext2 = fmaf(head.ext[c], head.ext[c], ext2);
    }
    const float hl = __double2float_ru(__dmul_rn(h, il)) * (1.0f + 0x1p-18f);
    const int n_sub = (head.count + kDfSub - 1) / kDfSub;
    k.floor2 = fmaxf(hl * hl * (1.0f + 0x1p-18f), ext2 * 0x1p-8f);
    k.direct = 0;
    k.loose = 0;
    k.close = 0;
    k.rmin2 = 0x1p60f;
    if (!__all_sync(0xffffffffu, !live || at < kDfRange)) {
        k.direct = (1u << n_sub) - 1u;
        return k;
    }
    for (int q = 0; q < n_sub; ++q) {
        const float *box = tile + kDfHeader + 6 * q;
        float gap2 = 0.0f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float gap = fmaxf(box[c] - tg.h[c], tg.h[c] - box[3 + c]);
            gap = fmaxf(0.0f, fmaf(-0x1p-20f, fabsf(tg.h[c]) + 1.0f, gap));
            gap2 = fmaf(gap, gap, gap2);
        }
        gap2 *= 1.0f - 0x1p-18f;
        const float diag2 = df_diagonal2(box), thr2 = df_radius2(k, diag2);
        const float least2 = fmaxf(gap2, thr2 * (1.0f - 0x1p-10f));
        if (__any_sync(0xffffffffu, live && least2 < kDfLeast2)) {
            k.direct |= 1u << q;
            continue;
        }
        if (__any_sync(0xffffffffu, live && !(gap2 > thr2))) {
            // (mostly softened pairs: no list)
            if (hl * hl > 0.25f * diag2) {
                k.direct |= 1u << q;
                continue;
            }
            if (LOOSE) {
                const int real = min(kDfSub, head.count - kDfSub * q);
                const int near = __reduce_add_sync(0xffffffffu, live ? df_count_close<S>(tile, q, real, tg, thr2) : 0);
                if ((float)near > kDfLoose * (float)(real * __popc(__ballot_sync(0xffffffffu, live)))) {
                    k.direct |= 1u << q;
                    k.loose |= 1u << q;
                    continue;
                }
            }
            k.close |= 1u << q;
        }
        // (lanes without a target: any window)
        if (live) k.rmin2 = fminf(k.rmin2, least2);
    }
    return k;
}

// The target's offset from a tile's centre in units of L.
__device__ __forceinline__ double df_offset(const DfHead &head, const double c[3], const double x[3],
                                            DfTarget &tg)
{
    const double il = pow2d(-head.el);
    const double xs[3] = {__dmul_rn(__dsub_rn(x[0], c[0]), il), __dmul_rn(__dsub_rn(x[1], c[1]), il),
                          __dmul_rn(__dsub_rn(x[2], c[2]), il)};
    df_split(xs, tg);
    return il;
}

}  // namespace grav
