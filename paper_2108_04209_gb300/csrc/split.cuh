// FP64 sums of w_j / (d_j - x) on the FP32 pipe, and the products and sums of
// squares of zhat and b (below).
//
// The GB300 retires about 2 FP64 operations per clock and SM against 128 FP32
// ones, so a near-field term of the secular sweeps (7 FP64 instructions, 112
// cycles of the FP64 pipe per warp) is split into FP32 parts that keep the
// accuracy of the FP64 term:
//   * positions are 96-bit fixed-point numbers relative to the first pole,
//     scaled so that the problem's spread is at most 1 (weight of the last bit
//     2^-94), cut into four 24-bit parts that are exact floats.  The parts of
//     two positions subtract exactly, so a difference t = d_j - x is known to
//     2^-94 of the spread however close the two are: relative error 2^-52 at half
//     the smallest pole gap accepted (2^-41 of the spread);
//   * t is summed into two floats, the reciprocal is a corrected MUFU seed and
//     its residual (relative error ~2^-47), the product with the weight (two
//     floats) another two floats;
//   * terms are added by error-free FP32 additions in blocks of 32 (renormalised
//     every 8), the blocks' sums likewise: an error of ~2^-47 of the sum.
// The FP64 form it replaces takes one Newton step from a 2^-22 seed (relative
// error up to 2^-44 per term, always of one sign); see rcp_nr1.
//
// The two poles next to a root (one is its origin: t = -y exactly, y of any
// size), which carry most of its sum, are left out of the FP32 sum and added by
// the caller in FP64.  Problems whose poles are closer
// than 2^-41 of the spread, or whose spread or weights leave the exponent range,
// keep the FP64 sweep.
//
// Measured (GB300, 4096 problems of 32..2048 poles): near-field sweeps of the
// FMM problems 36.1 -> 10.1 ms, their tail pass 4.8 -> 2.3, direct sweeps 13.2
// -> 1.45, zhat 4.9 + 1.1 -> 2.4 + 0.6, b 7.0 + 1.7 -> 2.0 + 0.5 ms (FMM +
// direct); with the far fields' series and steps of Root::update_split 5.2, 0.9
// and 1.3 ms for the three sweeps.  Against quadruple precision: roots' gaps as before (median 4e-15
// relative below 500 poles), zhat 7e-16 -> 9e-17 and b 3e-16 -> 9e-17 (rms,
// direct problems).
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define FF_HD __host__ __device__ __forceinline__
#else
#define FF_HD inline
#endif

// rounded FP32 operations that the compiler must not contract
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float ff_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float ff_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float ff_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float ff_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float ff_rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ int64_t ff_bits(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ double ff_double(int64_t b) { return __longlong_as_double(b); }
#else
#include <math.h>
#include <string.h>
FF_HD float ff_add(float a, float b) { volatile float r = a + b; return r; }
FF_HD float ff_sub(float a, float b) { volatile float r = a - b; return r; }
FF_HD float ff_mul(float a, float b) { volatile float r = a * b; return r; }
FF_HD float ff_fma(float a, float b, float c) { return fmaf(a, b, c); }
FF_HD float ff_rcp(float x) { return 1.0f / x; }      // the MUFU is within one unit of it
FF_HD int64_t ff_bits(double v) { int64_t b; memcpy(&b, &v, 8); return b; }
FF_HD double ff_double(int64_t b) { double v; memcpy(&v, &b, 8); return v; }
#endif

struct alignas(16) ff_f4 { float x, y, z, w; };
struct alignas(8) ff_f2 { float x, y; };

FF_HD int ff_exp(double v) { return (int)((ff_bits(v) >> 52) & 0x7FF); }
FF_HD double ff_pow2(int e) { return ff_double((int64_t)(e + 1023) << 52); }      // -1022 <= e <= 1023

// Scale of one problem: positions times 2^kk, weights times 2^-kw.
struct FfScale {
    __int128 ref;         // fixed-point position of the first pole
    int kk, kw;
    bool ok;              // spread and total weight in the exponent range
};

// v 2^(kk + 94) rounded toward zero, modulo 2^128 (differences of positions
// within the spread are at most 2^94, so the modulus does not show)
FF_HD __int128 ff_fixed(double v, int kk)
{
    const int64_t b = ff_bits(v);
    const int e = (int)((b >> 52) & 0x7FF);
    const uint64_t mant = (e == 0) ? 0ull : (((uint64_t)b & 0xFFFFFFFFFFFFFull) | (1ull << 52));
    const int s = e - 1075 + 94 + kk;
    unsigned __int128 m = 0;
    if (s >= 0) {
        if (s < 128) m = (unsigned __int128)mant << s;
    } else if (s > -64) {
        m = mant >> (-s);
    }
    return (b < 0) ? -(__int128)m : (__int128)m;
}

// d0, d1: first and last pole, w: sum of the weights
FF_HD FfScale ff_scale(double d0, double d1, double w)
{
    FfScale s;
    const int eh = ff_exp(d1 - d0), ew = ff_exp(w);
    s.ok = eh > 723 && eh < 1323 && ew > 723 && ew < 1323 && ff_exp(d0) < 1323 && ff_exp(d1) < 1323;
    s.kk = -(eh - 1023 + 1);
    s.kw = ew - 1023 + 1;
    s.ref = s.ok ? ff_fixed(d0, s.kk) : 0;
    return s;
}

// smallest distance of neighbouring poles that the fixed-point parts resolve
FF_HD bool ff_gap_ok(double da, double db, int kk) { return db - da >= ff_pow2(-kk - 41); }

// four 24-bit parts of a position relative to the first pole
FF_HD ff_f4 ff_parts(__int128 v)
{
    ff_f4 p;
    p.x = (float)(int)(v >> 72) * 0x1p-22f;
    p.y = (float)((unsigned)(v >> 48) & 0xFFFFFFu) * 0x1p-46f;
    p.z = (float)((unsigned)(v >> 24) & 0xFFFFFFu) * 0x1p-70f;
    p.w = (float)((unsigned)v & 0xFFFFFFu) * 0x1p-94f;
    return p;
}

FF_HD ff_f4 ff_pole(double d, const FfScale &s) { return ff_parts(ff_fixed(d, s.kk) - s.ref); }
FF_HD ff_f4 ff_point(double dK, double y, const FfScale &s)
{
    return ff_parts(ff_fixed(dK, s.kk) + ff_fixed(y, s.kk) - s.ref);
}
FF_HD ff_f2 ff_weight(double w, int kw)
{
    const double ws = w * ff_pow2(-kw);
    ff_f2 p;
    p.x = (float)ws;
    p.y = (float)(ws - (double)p.x);
    return p;
}

// t = d - x in two floats: the leading parts cancel exactly when they agree,
// so every FastTwoSum below meets |first| >= |second| or first = 0
FF_HD void ff_diff(const ff_f4 &d, const ff_f4 &x, float &t, float &tl)
{
    const float a = ff_sub(d.x, x.x), b = ff_sub(d.y, x.y), c = ff_sub(d.z, x.z), e = ff_sub(d.w, x.w);
    const float s = ff_add(a, b);
    const float u = ff_add(ff_sub(b, ff_sub(s, a)), c);
    t = ff_add(s, u);
    tl = ff_add(ff_sub(u, ff_sub(t, s)), e);
}

// p + pl = w / (d - x), q ~ w / (d - x)^2
FF_HD void ff_term(const ff_f4 &d, const ff_f2 &w, const ff_f4 &x, float &p, float &pl, float &q)
{
    float t, tl;
    ff_diff(d, x, t, tl);
    float r = ff_rcp(t);
    r = ff_fma(r, ff_fma(-t, r, 1.0f), r);
    const float rl = ff_mul(r, ff_fma(-tl, r, ff_fma(-t, r, 1.0f)));
    p = ff_mul(w.x, r);
    pl = ff_fma(w.y, r, ff_fma(w.x, rl, ff_fma(w.x, r, -p)));
    q = ff_mul(p, r);
}

// p + pl = w / (t + tl)
FF_HD void ff_div(const ff_f2 &w, float t, float tl, float &p, float &pl)
{
    float r = ff_rcp(t);
    r = ff_fma(r, ff_fma(-t, r, 1.0f), r);
    const float rl = ff_mul(r, ff_fma(-tl, r, ff_fma(-t, r, 1.0f)));
    p = ff_mul(w.x, r);
    pl = ff_fma(w.y, r, ff_fma(w.x, rl, ff_fma(w.x, r, -p)));
}

// p + pl = w / (d - x)^2
FF_HD void ff_term2(const ff_f4 &d, const ff_f2 &w, const ff_f4 &x, float &p, float &pl)
{
    float t, tl;
    ff_diff(d, x, t, tl);
    float r = ff_rcp(t);
    r = ff_fma(r, ff_fma(-t, r, 1.0f), r);
    const float rl = ff_mul(r, ff_fma(-tl, r, ff_fma(-t, r, 1.0f)));
    const float a = ff_mul(w.x, r);
    const float al = ff_fma(w.y, r, ff_fma(w.x, rl, ff_fma(w.x, r, -a)));
    p = ff_mul(a, r);
    pl = ff_fma(al, r, ff_fma(a, rl, ff_fma(a, r, -p)));
}

// running sums of one root: s + sl (+ c, see ff_close3) of all terms (b + bl of the
// current block), psi of the terms at and below the root's index (only for the stopping test's
// scale and the step's model), and the two derivative sums of the model, in
// single precision
struct FfAcc { float s, sl, c, b, bl, psi, dpsi, dphi; };

FF_HD void ff_addto(FfAcc &A, float p, float pl)
{
    const float s = ff_add(A.b, p);
    const float v = ff_sub(s, A.b);
    const float err = ff_add(ff_sub(A.b, ff_sub(s, v)), ff_sub(p, v));
    A.b = s;
    A.bl = ff_add(A.bl, ff_add(err, pl));
}

FF_HD void ff_norm(FfAcc &A)
{
    const float s = ff_add(A.b, A.bl);
    A.bl = ff_sub(A.bl, ff_sub(s, A.b));
    A.b = s;
}

// the block's sum into the total; the next block starts at zero
FF_HD void ff_close(FfAcc &A)
{
    ff_norm(A);
    const float s = ff_add(A.s, A.b);
    const float v = ff_sub(s, A.s);
    const float err = ff_add(ff_sub(A.s, ff_sub(s, v)), ff_sub(A.b, v));
    const float l = ff_add(A.sl, ff_add(err, A.bl));
    A.s = ff_add(s, l);
    A.sl = ff_sub(l, ff_sub(A.s, s));
    A.b = A.bl = 0.0f;
}

// The same with a total of three floats, for sums of many blocks: in two, every close
// rounds it at 2^-50, which over 4000 poles or the 80 box pairs of a far field is
// more than the terms' own errors leave (median error of the roots' gaps, 4000
// poles, direct sums: 9e-15 so, 7.7e-15 with three, 6.6e-15 by FP64 sums)
FF_HD void ff_close3(FfAcc &A)
{
    ff_norm(A);
    const float s = ff_add(A.s, A.b);
    const float v = ff_sub(s, A.s);
    const float err = ff_add(ff_sub(A.s, ff_sub(s, v)), ff_sub(A.b, v));
    const float t = ff_add(err, A.bl);
    const float v1 = ff_sub(t, err);
    const float e1 = ff_add(ff_sub(err, ff_sub(t, v1)), ff_sub(A.bl, v1));
    const float l = ff_add(A.sl, t);
    const float v2 = ff_sub(l, A.sl);
    const float e2 = ff_add(ff_sub(A.sl, ff_sub(l, v2)), ff_sub(t, v2));
    A.c = ff_add(A.c, ff_add(e1, e2));
    A.s = ff_add(s, l);
    A.sl = ff_sub(l, ff_sub(A.s, s));
    A.b = A.bl = 0.0f;
}

// the third part into the second, once all blocks are in
FF_HD void ff_fold(FfAcc &A)
{
    A.sl = ff_add(A.sl, A.c);
    A.c = 0.0f;
}

// another part's sums of the same root into A (the same result either way round)
FF_HD void ff_merge(FfAcc &A, float s, float sl, float psi, float dpsi, float dphi)
{
    const float t = ff_add(A.s, s);
    const float v = ff_sub(t, A.s);
    const float l = ff_add(ff_add(ff_sub(A.s, ff_sub(t, v)), ff_sub(s, v)), ff_add(A.sl, sl));
    A.s = ff_add(t, l);
    A.sl = ff_sub(l, ff_sub(A.s, t));
    A.psi += psi;
    A.dpsi += dpsi;
    A.dphi += dphi;
}

// the term of pole j when it may lie on either side of root k; the two next to
// the root are left out
FF_HD void ff_select(FfAcc &A, float p, float pl, float q, int j, int k)
{
    const bool next = (unsigned)(j - k) <= 1u, left = j < k;
    p = next ? 0.0f : p;
    pl = next ? 0.0f : pl;
    q = next ? 0.0f : q;
    ff_addto(A, p, pl);
    A.psi += left ? p : 0.0f;
    A.dpsi += left ? q : 0.0f;
    A.dphi += left ? 0.0f : q;
}

// Terms j0 .. j1-1 of staged poles whose first has index jg0 in the problem.
// k is the root's index; the warp's roots have indices kwlo .. kwhi, so only
// kwlo .. kwhi+1 need the per-root side.  LONG: more than a few blocks in all.
template <bool LONG = true>
FF_HD void ff_sweep(const ff_f4 *sd, const ff_f2 *sw, int j0, int j1, int jg0, int k, int kwlo, int kwhi,
                    const ff_f4 &x, FfAcc &A)
{
    int ea = kwlo - jg0, eb = kwhi + 2 - jg0;
    ea = ea < j0 ? j0 : (ea > j1 ? j1 : ea);
    eb = eb < ea ? ea : (eb > j1 ? j1 : eb);
    float p, pl, q;
    for (int c = j0; c < ea; c += 32) {
        const int e = c + 32 < ea ? c + 32 : ea;
        int j = c;
        for (; j + 8 <= e; j += 8) {
#pragma unroll
            for (int i = 0; i < 8; i++) {
                ff_term(sd[j + i], sw[j + i], x, p, pl, q);
                ff_addto(A, p, pl);
                A.dpsi += q;
            }
            ff_norm(A);
        }
        for (; j < e; j++) {
            ff_term(sd[j], sw[j], x, p, pl, q);
            ff_addto(A, p, pl);
            A.dpsi += q;
        }
        A.psi += A.b;
        if (LONG) ff_close3(A); else ff_close(A);
    }
    for (int c = ea; c < eb; c += 32) {
        const int e = c + 32 < eb ? c + 32 : eb;
        for (int j = c; j < e; j += 4) {
#pragma unroll
            for (int i = 0; i < 4; i++) {
                if (j + i >= e) break;
                ff_term(sd[j + i], sw[j + i], x, p, pl, q);
                ff_select(A, p, pl, q, jg0 + j + i, k);
            }
            ff_norm(A);
        }
        if (LONG) ff_close3(A); else ff_close(A);
    }
    for (int c = eb; c < j1; c += 32) {
        const int e = c + 32 < j1 ? c + 32 : j1;
        int j = c;
        for (; j + 8 <= e; j += 8) {
#pragma unroll
            for (int i = 0; i < 8; i++) {
                ff_term(sd[j + i], sw[j + i], x, p, pl, q);
                ff_addto(A, p, pl);
                A.dphi += q;
            }
            ff_norm(A);
        }
        for (; j < e; j++) {
            ff_term(sd[j], sw[j], x, p, pl, q);
            ff_addto(A, p, pl);
            A.dphi += q;
        }
        if (LONG) ff_close3(A); else ff_close(A);
    }
    if (LONG) ff_fold(A);
}

// ---------------------------------------------------------------------------
// Three floats (a + b + c, |b| <= ulp(a)/2 or so): b and zhat need the accuracy
// of FP64 in every term (relative error below 2^-60 here, against 2^-53), and an
// FP64 operation costs the issue slots of 64 FP32 ones.
// ---------------------------------------------------------------------------
struct ff_t3 { float a, b, c; };

FF_HD void ff_two_sum(float x, float y, float &s, float &e)
{
    s = ff_add(x, y);
    const float v = ff_sub(s, x);
    e = ff_add(ff_sub(x, ff_sub(s, v)), ff_sub(y, v));
}

FF_HD void ff_fast_sum(float x, float y, float &s, float &e)      // |x| >= |y| or x = 0
{
    s = ff_add(x, y);
    e = ff_sub(y, ff_sub(s, x));
}

FF_HD void ff_two_mul(float x, float y, float &p, float &e)
{
    p = ff_mul(x, y);
    e = ff_fma(x, y, -p);
}

// d - x: exact up to the last part's rounding (see ff_diff; the errors of the
// two leading sums are multiples of 2^-70 and larger than what follows)
FF_HD ff_t3 ff_diff3(const ff_f4 &d, const ff_f4 &x)
{
    const float a = ff_sub(d.x, x.x), b = ff_sub(d.y, x.y), c = ff_sub(d.z, x.z), e = ff_sub(d.w, x.w);
    float s, r, u, v, u2;
    ff_t3 t;
    ff_fast_sum(a, b, s, r);
    ff_fast_sum(r, c, u, v);
    ff_fast_sum(s, u, t.a, u2);
    ff_fast_sum(u2, ff_add(v, e), t.b, t.c);
    return t;
}

FF_HD ff_t3 ff_mul3(const ff_t3 &x, const ff_t3 &y)
{
    float p, e1, q, e2, r, e3, s, f, b, g;
    ff_two_mul(x.a, y.a, p, e1);
    ff_two_mul(x.a, y.b, q, e2);
    ff_two_mul(x.b, y.a, r, e3);
    ff_two_sum(q, r, s, f);
    ff_two_sum(e1, s, b, g);
    const float c = ff_fma(x.a, y.c, ff_fma(x.c, y.a, ff_fma(x.b, y.b, ff_add(ff_add(e2, e3), ff_add(f, g)))));
    ff_t3 o;
    ff_fast_sum(p, b, o.a, s);
    ff_fast_sum(s, c, o.b, o.c);
    return o;
}

// 1 / t: with the seed r, 1 - t r = e exactly in two floats, 1/t = r (1 + e + e^2)
FF_HD ff_t3 ff_rcp3(const ff_t3 &t)
{
    const float r = ff_rcp(t.a);
    float p, pe, q, qe, h, hl, e, el, k, ke;
    ff_two_mul(t.a, r, p, pe);
    ff_two_mul(t.b, r, q, qe);
    ff_two_sum(pe, q, h, hl);
    ff_two_sum(ff_sub(1.0f, p), -h, e, el);
    el = ff_sub(el, ff_add(hl, ff_fma(t.c, r, qe)));
    el = ff_fma(e, e, el);
    ff_two_mul(r, e, k, ke);
    ff_t3 o;
    ff_fast_sum(r, k, o.a, h);
    ff_fast_sum(h, ff_fma(r, el, ke), o.b, o.c);
    return o;
}

FF_HD ff_t3 ff_sqr3(const ff_t3 &x)
{
    float p, e1, q, e2, b, g;
    const float x2 = x.a + x.a;
    ff_two_mul(x.a, x.a, p, e1);
    ff_two_mul(x2, x.b, q, e2);
    ff_two_sum(e1, q, b, g);
    ff_t3 o;
    ff_fast_sum(p, b, o.a, e1);
    ff_fast_sum(e1, ff_fma(x2, x.c, ff_fma(x.b, x.b, ff_add(e2, g))), o.b, o.c);
    return o;
}

// s += x (no renormalisation of s.b, s.c: they stay a few ulps of s.a)
FF_HD void ff_acc3(ff_t3 &s, const ff_t3 &x)
{
    float e, f, g;
    ff_two_sum(s.a, x.a, s.a, e);
    ff_two_sum(x.b, e, e, f);
    ff_two_sum(s.b, e, s.b, g);
    s.c = ff_add(s.c, ff_add(ff_add(f, g), x.c));
}

// p *= 1 + x
FF_HD void ff_mul1p3(ff_t3 &p, const ff_t3 &x)
{
    const ff_t3 k = ff_mul3(p, x);
    ff_acc3(p, k);
    float s, e;
    ff_fast_sum(p.a, p.b, s, e);
    p.a = s;
    ff_fast_sum(e, p.c, p.b, p.c);
}

// an FP64 value (scaled into range by the caller) as three floats, exactly
FF_HD ff_t3 ff_split3(double v)
{
    ff_t3 t;
    t.a = (float)v;
    const double r = v - (double)t.a;
    t.b = (float)r;
    t.c = (float)(r - (double)t.b);
    return t;
}

FF_HD double ff_join3(const ff_t3 &t) { return ((double)t.c + (double)t.b) + (double)t.a; }

// ---------------------------------------------------------------------------
// Products of differences by integers (zhat, eq. (4.23)): a 64-bit mantissa and
// an exponent.  A difference of two 96-bit positions is exact, its leading 64
// bits keep it to 2^-63, and a product costs one 64-bit high multiply.
// ---------------------------------------------------------------------------
struct ff_u96 { unsigned lo, mid, hi; };          // position relative to the first pole, two's complement

struct FfProd { uint64_t m; int e; };             // m 2^e, m normalised by ff_prod_norm

FF_HD int ff_clz(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}

FF_HD uint64_t ff_mulhi(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

FF_HD void ff_prod_norm(FfProd &p)
{
    const int c = ff_clz(p.m);
    p.m <<= c;
    p.e -= c;
}

// p *= |x - y| (in units of the positions' last bit); use = false leaves p.
// Between two normalisations at most 8 factors (one bit each is lost).
FF_HD void ff_prod_mul(FfProd &p, const ff_u96 &x, const ff_u96 &y, bool use)
{
    // x - y over three words, its absolute value
    const uint64_t xl = ((uint64_t)x.mid << 32) | x.lo, yl = ((uint64_t)y.mid << 32) | y.lo;
    uint64_t l = xl - yl;
    unsigned h = x.hi - y.hi - (xl < yl ? 1u : 0u);
    if ((int)h < 0) {
        h = ~h + (l == 0 ? 1u : 0u);
        l = 0ull - l;
    }
    // leading 64 bits
    int e = 32;
    uint64_t t = ((uint64_t)h << 32) | (l >> 32);
    unsigned rest = (unsigned)l;
    if (t >> 32 == 0) { t = (t << 32) | rest; rest = 0; e = 0; }
    const int c = ff_clz(t);
    t = (t << (c & 63)) | (c > 0 && c < 32 ? rest >> (32 - c) : 0u);
    e -= c;
    const uint64_t q = ff_mulhi(p.m, t);
    p.m = use ? q : p.m;
    p.e = use ? p.e + e + 64 : p.e;
}

// positions as words for ff_prod_mul (16 bytes: one vector load)
struct alignas(16) ff_w4 { unsigned lo, mid, hi, pad; };
FF_HD ff_w4 ff_words4(__int128 v)
{
    ff_w4 w;
    w.lo = (unsigned)v;
    w.mid = (unsigned)(v >> 32);
    w.hi = (unsigned)(v >> 64);
    w.pad = 0;
    return w;
}

// num *= prod |lambda_j - d_i|, den *= prod |d_j - d_i| over cnt staged sources
// (first index j0), without j = i and j = i - 1 (an eigenvalue next to d_i may
// be closer than the positions resolve: the caller adds those in FP64)
FF_HD void ff_prod_sweep(const ff_w4 *sd, const ff_w4 *sl, int cnt, int j0, int i, const ff_u96 &di, FfProd &num,
                         FfProd &den)
{
    for (int c = 0; c < cnt; c += 8) {
        const int e = c + 8 < cnt ? c + 8 : cnt;
#pragma unroll 2
        for (int j = c; j < e; j++) {
            const bool use = (unsigned)(i - (j0 + j)) > 1u;
            const ff_w4 a = sl[j], b = sd[j];
            const ff_u96 la = {a.lo, a.mid, a.hi}, db = {b.lo, b.mid, b.hi};
            ff_prod_mul(num, la, di, use);
            ff_prod_mul(den, db, di, use);
        }
        ff_prod_norm(num);
        ff_prod_norm(den);
    }
}

// S += sum (v_j / (d_j - x))^2 over cnt staged sources (first index j0),
// without j = K (t = -eta, added by the caller in FP64)
FF_HD void ff_sqr_sweep(const ff_f4 *sd, const ff_f4 *sv, int cnt, int j0, int K, const ff_f4 &x, ff_t3 &S)
{
#pragma unroll 2
    for (int j = 0; j < cnt; j++) {
        const ff_f4 v = sv[j];
        const ff_t3 v3 = {v.x, v.y, v.z};
        ff_t3 q = ff_sqr3(ff_mul3(v3, ff_rcp3(ff_diff3(sd[j], x))));
        const bool own = j0 + j == K;
        q.a = own ? 0.0f : q.a;
        q.b = own ? 0.0f : q.b;
        q.c = own ? 0.0f : q.c;
        ff_acc3(S, q);
    }
}

// ---------------------------------------------------------------------------
// log(t + tl), t > 0, in two floats (absolute error ~2^-47 for exponents e of a
// few): table-driven argument reduction (P. T. P. Tang, Table-driven
// implementation of the logarithm function, 1990): with c_i the reciprocal of
// the middle of the i-th of 128 intervals of [1, 2), rounded to 10 bits,
// m c_i - 1 = d is exact in two floats and log = e ln 2 - log c_i + log1p(d),
// the last by its Taylor series.  e0 is subtracted from the exponent.
// ---------------------------------------------------------------------------
struct ff_logtab { float c, h, l; };              // c_i and -log c_i

FF_HD float ff_logc(int i) { return rintf(512.0f / (1.0f + (i + 0.5f) / 128.0f)) * 0x1p-9f; }

FF_HD int ff_fexp(float t)
{
#ifdef __CUDA_ARCH__
    return (__float_as_int(t) >> 23) - 127;
#else
    int b;
    memcpy(&b, &t, 4);
    return (b >> 23) - 127;
#endif
}

FF_HD void ff_log(float t, float tl, int e0, const ff_logtab *tab, float &y, float &yl)
{
    const float LN2H = 0x1.62e43000p-1f, LN2L = -0x1.05c61000p-29f;      // ln 2
    const int e = ff_fexp(t);
#ifdef __CUDA_ARCH__
    const int b = __float_as_int(t);
    const float m = __int_as_float((b & 0x7FFFFF) | 0x3F800000), sc = __int_as_float((127 - e) << 23);
#else
    int b;
    memcpy(&b, &t, 4);
    const float m = ldexpf(t, -e), sc = ldexpf(1.0f, -e);
#endif
    const ff_logtab T = tab[(b >> 16) & 127];
    float p, pe, d, dl, s, sl, a, al;
    ff_two_mul(m, T.c, p, pe);
    ff_fast_sum(ff_sub(p, 1.0f), ff_fma(ff_mul(tl, sc), T.c, pe), d, dl);
    const float q = ff_mul(d, d), qe = ff_fma(d + d, dl, ff_fma(d, d, -q));
    float r = ff_fma(d, 1.0f / 7.0f, -1.0f / 6.0f);
    r = ff_fma(d, r, 0.2f);
    r = ff_fma(d, r, -0.25f);
    r = ff_mul(ff_mul(d, q), ff_fma(d, r, 1.0f / 3.0f));
    ff_fast_sum(d, -0.5f * q, s, sl);
    sl = ff_add(sl, ff_add(ff_fma(-0.5f, qe, dl), r));
    ff_two_sum(T.h, s, a, al);
    al = ff_add(al, ff_add(T.l, sl));
    const float k = (float)(e - e0);
    ff_two_mul(k, LN2H, p, pe);
    ff_two_sum(p, a, y, yl);
    yl = ff_add(yl, ff_add(ff_fma(k, LN2L, pe), al));
}
