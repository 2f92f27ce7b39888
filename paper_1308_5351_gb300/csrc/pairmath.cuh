// Per-pair arithmetic shared by the pair-sum kernels (device code only).
#pragma once

#include <cuda_runtime.h>

namespace gnk {

// ------------------------------------------------------------------ reciprocal
static __device__ __forceinline__ double rcp_seed_f64(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}

// 1/x in full FP64 from the hardware seed y0 (relative error below 2^-19):
// with e = 1 - x y0 we have 1/x = y0 / (1 - e) = y0 (1 + e + e^2 + ...), so
// y0 (1 + e + e^2) leaves the relative error e^3 < 2^-57, below half an ulp
// after rounding for all but a vanishing set of inputs.
static __device__ __forceinline__ double recip_f64(double x) {
    const double y0 = rcp_seed_f64(x);
    const double e = fma(-x, y0, 1.0);
    const double t = fma(e, e, e);
    return fma(y0, t, y0);
}

static __device__ __forceinline__ float recip_f32(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ------------------------------------------------------------------ double-float (df32)
// FP64-class Cauchy sums on the FP32 pipe.  A df32 number is an unevaluated
// sum hi + lo of two floats (about 48 significant bits).  Error-free
// transformations (Knuth's TwoSum, Dekker's product via FMA) carry the
// rounding errors of every step; positions are taken relative to the source
// tile's FP64 reference node (each target forms its offset in FP64 once per
// tile), so the difference of two nearby nodes keeps its leading bits.  Per
// pair: ~22 flops for d, 16 for |d|^2, 3 for the reciprocal (one Newton step
// from rcp.approx), 8 for 1/d, 16 for the four weight products and 32 for
// the two compensated accumulations, all on the FP32 pipe.
struct df {
    float h, l;
};

// The _rn intrinsics are never contracted into FMAs by the compiler, which
// the error-free transformations below rely on.
static __device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

static __device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}

// a - b for df32 operands (Bailey's add with a final renormalisation)
static __device__ __forceinline__ df df_sub(float ah, float al, float bh, float bl) {
    float s, e;
    two_sum(ah, -bh, s, e);
    e = __fadd_rn(e, __fsub_rn(al, bl));
    df r;
    fast_two_sum(s, e, r.h, r.l);
    return r;
}

// product of two df32 values, unnormalised (hi = fl(a.h b.h), lo = error + cross terms)
static __device__ __forceinline__ df df_mul(df a, df b) {
    df r;
    r.h = __fmul_rn(a.h, b.h);
    float e = fmaf(a.h, b.h, -r.h);
    e = fmaf(a.h, b.l, e);
    e = fmaf(a.l, b.h, e);
    r.l = e;
    return r;
}

// acc += p (compensated: the hi sum's rounding error goes to acc.l)
static __device__ __forceinline__ void df_acc(df& acc, df p) {
    float s, e;
    two_sum(acc.h, p.h, s, e);
    acc.h = s;
    acc.l = __fadd_rn(acc.l, __fadd_rn(e, p.l));
}

static __device__ __forceinline__ df df_split(double v) {
    df r;
    r.h = (float)v;
    r.l = (float)(v - (double)r.h);
    return r;
}

// df_split without the FP64 pipe (each conversion there is a 64-cycle
// dependent step on GB300): from the bits of v, hi = v truncated to 24
// significant bits (exact as a float) and lo = the next 23 bits, so
// |v - (hi + lo)| < 2^-46 |v|.  For 2^-80 <= |v| < 2^101; zero, tiny, huge and
// non-finite values take df_split.
// (out of line, so that the compiler branches to it instead of evaluating its
// FP64 conversions beside every fast split)
static __device__ __noinline__ df df_split_slow(double v) { return df_split(v); }

static __device__ __forceinline__ df df_split_fast(double v) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const unsigned hi = (unsigned)(bits >> 32), lo = (unsigned)bits;
    const unsigned e = (hi >> 20) & 0x7ffu;  // biased exponent
    if (e - 943u > 180u) return df_split_slow(v);
    const unsigned sign = hi & 0x80000000u;
    df r;
    r.h = __uint_as_float(sign | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
    // the low 29 bits of the significand: their top 23 exactly through the 2^23
    // bias, scaled by 2^(e - 1069)
    const float m = __fsub_rn(__uint_as_float(0x4b000000u | ((lo & 0x1fffffffu) >> 6)), 8388608.0f);
    r.l = __uint_as_float(__float_as_uint(__fmul_rn(m, __uint_as_float((e - 942u) << 23))) | sign);
    return r;
}

// ------------------------------------------------------------------ packed double-float
// Two independent double-float values per float2 (lane x, lane y) with the
// sm_100 packed FP32 intrinsics: one instruction issues both lanes, so the
// FP32 pipe rather than instruction issue bounds the kernels.  The _rn forms
// are never contracted.  Subtraction is written as an FMA with -1, which is
// exact and rounds once like a subtraction.
struct df2 {
    float2 h, l;
};

static __device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
static __device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
static __device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
static __device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
static __device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
static __device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.0f), a); }

static __device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
    s = add2(a, b);
    const float2 bb = sub2(s, a);
    e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

static __device__ __forceinline__ void two_diff2(float2 a, float2 b, float2& s, float2& e) {
    s = sub2(a, b);
    const float2 bb = sub2(s, a);
    e = sub2(sub2(a, sub2(s, bb)), add2(b, bb));
}

// a - b, b the same for both lanes (Bailey's add, renormalised)
static __device__ __forceinline__ df2 df2_sub(float2 ah, float2 al, float2 bh, float2 bl) {
    float2 s, e;
    two_diff2(ah, bh, s, e);
    e = add2(e, sub2(al, bl));
    df2 r;
    r.h = add2(s, e);
    r.l = sub2(e, sub2(r.h, s));
    return r;
}

static __device__ __forceinline__ df2 df2_mul(df2 a, df2 b) {
    df2 r;
    r.h = mul2(a.h, b.h);
    float2 e = fma2(a.h, b.h, neg2(r.h));
    e = fma2(a.h, b.l, e);
    e = fma2(a.l, b.h, e);
    r.l = e;
    return r;
}

static __device__ __forceinline__ void df2_acc(df2& acc, df2 p) {
    float2 s, e;
    two_sum2(acc.h, p.h, s, e);
    acc.h = s;
    acc.l = add2(acc.l, add2(e, p.l));
}

static __device__ __forceinline__ void df2_dec(df2& acc, df2 p) {
    float2 s, e;
    two_diff2(acc.h, p.h, s, e);
    acc.h = s;
    acc.l = sub2(acc.l, sub2(p.l, e));
}

// ------------------------------------------------------------------ 1/d in FP64, on the FP32 pipe
// conj(d) / |d|^2 = ar - i ai of an FP64 difference d = dx + i dy, to FP64 accuracy,
// with no FP64 instruction: GB300's FP64 pipe (2 lanes per SM) bounds the FP64 pair
// kernels, and |d|^2, its reciprocal and the two products were 7 of the 13 to 17
// instructions of a pair there; the 220 instructions below take the 128 FP32
// lanes a third of the time that those 7 took.  dx and dy are split exactly into
// three floats (24 + 23 + 6 bits), |d|^2, its reciprocal and the products are
// formed as three-float sums with error-free transformations (relative error
// below 2^-60), and each result is rounded once to FP64 by integer arithmetic on
// its bits.  The error is below 1.01 ulp of the larger part, 0.51 away from powers
// of two (20 million pairs emulated against extended precision; the FP64
// sequence, with a rounding per step, reaches 2).  For 2^-40 <= max(|dx|, |dy|) < 2^40 with
// the smaller one zero or at least 2^-70; other pairs (and d = 0) take the FP64
// sequence, out of line so that the compiler branches to it.
static __device__ __noinline__ double2 inv_slow_f64(double dx, double dy) {
    const double inv = recip_f64(fma(dx, dx, dy * dy));
    return make_double2(dx * inv, dy * inv);
}

// v = h + m + l exactly (0 where v = 0); e: biased exponent of v, at least 949 or 0
static __device__ __forceinline__ void split3_bits(double v, float& h, float& m, float& l, unsigned& e) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    e = (hi >> 20) & 0x7ffu;
    const unsigned sign = hi & 0x80000000u;
    const bool nz = e != 0u;
    h = __uint_as_float(nz ? (sign | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29)) : 0u);
    const float sc = __uint_as_float(nz ? ((e - 948u) << 23) | sign : 0u);  // 2^(e - 1075)
    m = __fmul_rn(__fsub_rn(__uint_as_float(0x4b000000u | ((lo & 0x1fffffffu) >> 6)), 8388608.0f), __fmul_rn(sc, 64.0f));
    l = __fmul_rn(__fsub_rn(__uint_as_float(0x4b000000u | (lo & 63u)), 8388608.0f), sc);
}

// (h + m + l)(y0 + y1 + y2), rounded to FP64; |h y0| below 2^-75 keeps its leading float
static __device__ __forceinline__ double mul3_f64(float h, float m, float l, float y0, float y1, float y2) {
    float p = __fmul_rn(h, y0);
    const float pe = fmaf(h, y0, -p);
    const float u = __fmul_rn(h, y1), ue = fmaf(h, y1, -u);
    const float v = __fmul_rn(m, y0), ve = fmaf(m, y0, -v);
    float w, we, mid, me;
    two_sum(u, v, w, we);
    two_sum(w, pe, mid, me);
    fast_two_sum(p, mid, p, mid);  // |mid| at most half a unit of p's last place
    const float low = __fadd_rn(__fadd_rn(__fadd_rn(we, me), __fadd_rn(ue, ve)),
                                fmaf(h, y2, fmaf(m, y1, __fmul_rn(l, y0))));
    // p as FP64 bits, plus mid + low in units of its last place
    const unsigned f = __float_as_uint(p), ef = (f >> 23) & 255u;
    const float sc = __uint_as_float(ef >= 52u ? (306u - ef) << 23 : 0u);  // 2^(52 - (ef - 127))
    const float ms = __fmul_rn(mid, sc);                                  // at most 2^29
    const float tb = __fadd_rn(ms, 1610612736.0f);                        // 1.5 2^30: multiples of 128
    const float small = __fadd_rn(__fsub_rn(ms, __fsub_rn(tb, 1610612736.0f)), __fmul_rn(low, sc));
    const float ts = __fadd_rn(small, 12582912.0f);                       // 1.5 2^23: integers
    int di = ((__float_as_int(tb) - 0x4ec00000) << 7) + (__float_as_int(ts) - 0x4b400000);
    const int neg = (int)f >> 31;
    di = (di ^ neg) - neg;
    if ((f & 0x7fffffu) == 0u && di < 0) di += di;  // below a power of two the units are half
    const long long bits = (((long long)(f & 0x7fffffffu)) << 29) + (896LL << 52) + (long long)di;
    return __hiloint2double((int)((unsigned)(bits >> 32) | (f & 0x80000000u)), (int)bits);
}

static __device__ __forceinline__ void inv_conj_f64(double dx, double dy, double& ar, double& ai) {
    float hx, mx, lx, hy, my, ly;
    unsigned ex, ey;
    split3_bits(dx, hx, mx, lx, ex);
    split3_bits(dy, hy, my, ly, ey);
    const unsigned em = max(ex, ey);
    // (exponents, not comparisons of doubles, which would be FP64 instructions;
    // a denormal counts as zero)
    if (em - 983u >= 80u || ex - 1u < 952u || ey - 1u < 952u) {
        const double2 v = inv_slow_f64(dx, dy);
        ar = v.x;
        ai = v.y;
        return;
    }
    // |d|^2 = H + M + L
    const float ax = __fadd_rn(hx, hx), ay = __fadd_rn(hy, hy);
    const float p0x = __fmul_rn(hx, hx), e0x = fmaf(hx, hx, -p0x), p0y = __fmul_rn(hy, hy), e0y = fmaf(hy, hy, -p0y);
    const float p1x = __fmul_rn(ax, mx), e1x = fmaf(ax, mx, -p1x), p1y = __fmul_rn(ay, my), e1y = fmaf(ay, my, -p1y);
    const float rx = fmaf(ax, lx, __fmul_rn(mx, mx)), ry = fmaf(ay, ly, __fmul_rn(my, my));
    float H, t, s, u1, v, u2, M, u3, u4;
    two_sum(p0x, p0y, H, t);
    two_sum(p1x, p1y, s, u1);
    two_sum(e0x, e0y, v, u2);
    two_sum(s, v, M, u3);
    two_sum(M, t, M, u4);
    float L = __fadd_rn(__fadd_rn(__fadd_rn(u1, u2), __fadd_rn(u3, u4)), __fadd_rn(__fadd_rn(e1x, e1y), __fadd_rn(rx, ry)));
    fast_two_sum(H, M, H, M);
    fast_two_sum(M, L, M, L);
    // 1/|d|^2 = y0 (1 + e + e^2), e = 1 - (H + M + L) y0 to 2^-70
    const float y0 = recip_f32(H);
    const float tp = __fmul_rn(H, y0), te = fmaf(H, y0, -tp);
    const float mp = __fmul_rn(M, y0), me = fmaf(M, y0, -mp);
    float a, b, eh, c;
    two_sum(__fsub_rn(1.0f, tp), -te, a, b);
    two_sum(a, -mp, eh, c);
    const float sl = fmaf(eh, eh, __fsub_rn(__fadd_rn(b, c), fmaf(L, y0, me)));
    const float y1 = __fmul_rn(y0, eh), y2 = fmaf(y0, sl, fmaf(y0, eh, -y1));
    ar = mul3_f64(hx, mx, lx, y0, y1, y2);
    ai = mul3_f64(hy, my, ly, y0, y1, y2);
}

}  // namespace gnk
