// Device building blocks of the secular-equation solver shared by the
// direct tiled evaluator (rank1.cu) and the triangular FMM path (fmm.cu):
// the FP64 reciprocal, the bracketed quadratic root, the triangular sweep
// over staged poles (eqs. (4.7)-(4.10), shifted differences of eq. (4.14))
// and the per-root iteration state (Algorithm 2, stopping test eq. (4.12)).
#pragma once
#include "common.cuh"
#include "split.cuh"

namespace {

// ---------------------------------------------------------------------------
// FP64 reciprocal without the FP64 divide sequence.  The GB300 FP64 pipe
// retires ~2 DFMA per clock per SM, so every FP64 instruction of the inner
// loops counts, while integer and MUFU pipes are nearly free.  Seed: the
// leading 23 mantissa bits of |t| as a float in [1,2), reciprocal on the MUFU
// (rcp.approx.f32, relative error < 2^-22 after the truncation), exponent and
// sign rebuilt with integer arithmetic (valid for every normal double).  Then
// Newton-Raphson r <- r + r (1 - t r), which squares the relative error:
// one step -> < 2^-44, two steps -> correctly rounded up to ~1 ulp.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float mufu_rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ double rcp_seed(double t)
{
    const int hi = __double2hiint(t);
    const unsigned lo = (unsigned)__double2loint(t);
    const unsigned sign = (unsigned)hi & 0x80000000u;
    const int e = (hi >> 20) & 0x7FF;
    const unsigned mb = (((unsigned)hi & 0xFFFFFu) << 3) | (lo >> 29);
    const float rm = mufu_rcp(__uint_as_float(0x3F800000u | mb));   // in (0.5, 1]
    const unsigned rb = __float_as_uint(rm);
    const int E = (int)(rb >> 23) - 127 - (e - 1023) + 1023;
    const unsigned rmant = rb & 0x7FFFFFu;
    return __hiloint2double((int)(sign | ((unsigned)E << 20) | (rmant >> 3)), (int)(rmant << 29));
}

// one Newton step: relative error < 2^-44 (secular sweeps: every term of psi
// (phi) has the same sign, so the sum inherits the per-term bound, which is
// below the stopping tolerance of eq. (4.12) for m >= 32)
__device__ __forceinline__ double rcp_nr1(double t)
{
    double r = rcp_seed(t);
    double e = fma(-t, r, 1.0);
    return fma(r, e, r);
}

// full FP64 accuracy (b, Cauchy-like applications, the poles next to a root):
// one step of third order, r <- r + r (e + e^2) with e = 1 - t r below 2^-22
__device__ __forceinline__ double rcp_nr2(double t)
{
    const double r = rcp_seed(t);
    const double e = fma(-t, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// 1 / t, any t
__device__ __forceinline__ double rcp_any(double t)
{
    const int e = (__double2hiint(t) >> 20) & 0x7FF;
    return (e > 30 && e < 2016) ? rcp_nr2(t) : 1.0 / t;
}

// 1 / t rounded to nearest (Markstein, 1990: a reciprocal within an ulp, corrected
// by its residual)
__device__ __forceinline__ double rcp_rn(double t)
{
    const int e = (__double2hiint(t) >> 20) & 0x7FF;
    if (e < 31 || e > 2015) return 1.0 / t;
    const double r = rcp_nr2(t);
    return fma(r, fma(-t, r, 1.0), r);
}

// q^(-1/2) to about 2^-22 for a normal q > 0: the FP32 approximate reciprocal
// square root of the leading mantissa bits (scaled into [1, 4) to make the
// exponent even), the exponent halved by integer arithmetic; no conversion
// between FP64 and FP32 in the chain of dependent steps
__device__ __forceinline__ double rsqrt_seed(double q)
{
    const int hi = __double2hiint(q);
    const unsigned lo = (unsigned)__double2loint(q);
    const int e = ((hi >> 20) & 0x7FF) - 1023;
    const int odd = e & 1;
    const unsigned mb = (((unsigned)hi & 0xFFFFFu) << 3) | (lo >> 29);
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(((unsigned)(127 + odd) << 23) | mb)));
    const unsigned rb = __float_as_uint(r);                  // in (0.5, 1]
    const int E = (int)(rb >> 23) - 127 - (e - odd) / 2 + 1023;
    const unsigned rm = rb & 0x7FFFFFu;
    return __hiloint2double((int)(((unsigned)E << 20) | (rm >> 3)), (int)(rm << 29));
}

// q^(-1/2), one step of third order from the seed: with e = 1 - q y^2,
// y + y e (1/2 + 3/8 e)
__device__ __forceinline__ double rsqrt_nr(double q)
{
    const double y = rsqrt_seed(q);
    const double e = fma(-q * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

__device__ __forceinline__ double rsqrt_any(double q)
{
    const int h = __double2hiint(q), e = h >> 20;
    return (e > 30 && e < 2016) ? rsqrt_nr(q) : 1.0 / sqrt(q);
}

// sqrt(n / d 2^ex) = result 2^(ex / 2), ex made even; n and d of one sign
__device__ __forceinline__ double root_quot(double n, double d, int &ex)
{
    double q = n / d;
    if (ex & 1) { q *= 2.0; ex -= 1; }
    return sqrt(q);
}

// root of a*y^2 + b*y + c = 0 strictly inside (lo, hi), else the bracket middle
__device__ double quad_in(double a, double b, double c, double lo, double hi)
{
    double mid = 0.5 * (lo + hi);
    if (a == 0.0) {
        if (b == 0.0) return mid;
        double y = -c / b;
        return (y > lo && y < hi) ? y : mid;
    }
    double disc = b * b - 4.0 * a * c;
    if (!(disc >= 0.0)) return mid;
    double sq = sqrt(disc);
    double q = -0.5 * (b + (b >= 0 ? sq : -sq));
    double y1 = q / a;
    double y2 = (q != 0.0) ? c / q : y1;
    if (y1 > lo && y1 < hi) return y1;
    if (y2 > lo && y2 < hi) return y2;
    return mid;
}

// ---------------------------------------------------------------------------
// Secular roots.
// ---------------------------------------------------------------------------
struct Acc { double psi, phi, dpsi, dphi; };

// Accumulate the triangular parts over poles [j0, j1) of a staged chunk whose
// first pole has global index jg0.  Pole j goes to psi if j <= k, else to phi.
// The warp's roots are consecutive (kwlo..kwhi), so the loop runs in three
// warp-uniform regions; only the middle one selects per lane.
__device__ __forceinline__ int fexp(double v) { return (__double2hiint(v) >> 20) & 0x7FF; }

// Every term uses the shifted difference (d_j - d_K) - y of eq. (4.14).  (The
// local-shifting variant that takes d_j - x for far poles, eqs. (4.19)-(4.21),
// saves one FP64 subtraction per term but measured slower on GB300: the
// integer exponent test and branch cost more than the subtraction.)
__device__ __forceinline__ double shifted_t(double dj, double dK, double y)
{
    return (dj - dK) - y;
}

template <bool DERIV>
__device__ __forceinline__ void sweep(const double *__restrict__ sd, const double *__restrict__ sw,
                                      int j0, int j1, int jg0, int k, int kwlo, int kwhi,
                                      double dK, double y, Acc &A)
{
    // region A: global j <= kwlo -> psi for every lane
    int ea = min(j1, max(j0, kwlo - jg0 + 1));
#pragma unroll 4
    for (int j = j0; j < ea; j++) {
        double t = shifted_t(sd[j], dK, y);
        double r = rcp_nr1(t);
        if (DERIV) {
            double a = sw[j] * r;
            A.psi += a;
            A.dpsi = fma(a, r, A.dpsi);
        } else {
            A.psi = fma(sw[j], r, A.psi);
        }
    }
    // region B: kwlo < j <= kwhi -> per lane
    int eb = min(j1, max(ea, kwhi - jg0 + 1));
    for (int j = ea; j < eb; j++) {
        double t = shifted_t(sd[j], dK, y);
        double r = rcp_nr1(t);
        double a = sw[j] * r;
        if (jg0 + j <= k) { A.psi += a; if (DERIV) A.dpsi = fma(a, r, A.dpsi); }
        else              { A.phi += a; if (DERIV) A.dphi = fma(a, r, A.dphi); }
    }
    // region C: j > kwhi -> phi for every lane
#pragma unroll 4
    for (int j = eb; j < j1; j++) {
        double t = shifted_t(sd[j], dK, y);
        double r = rcp_nr1(t);
        if (DERIV) {
            double a = sw[j] * r;
            A.phi += a;
            A.dphi = fma(a, r, A.dphi);
        } else {
            A.phi = fma(sw[j], r, A.phi);
        }
    }
}

// v 2^k rounded to single precision (0 below its range, which the caller
// rules out above), by integer arithmetic: a conversion costs an FP64 slot
__device__ __forceinline__ float ff_top(double v, int k)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) + (1ull << 28);
    const int hi = (int)(b >> 32);
    const int e = ((hi >> 20) & 0x7FF) - 896 + k;
    const unsigned m = (unsigned)(b >> 29) & 0x7FFFFFu;
    return (e <= 0) ? 0.0f : __uint_as_float(((unsigned)hi & 0x80000000u) | ((unsigned)min(e, 254) << 23) | m);
}

// v 2^k in two floats (v 2^k a normal float or flushed to 0)
__device__ __forceinline__ ff_f2 ff_split2(double v, int k)
{
    const int hi = __double2hiint(v);
    const unsigned lo = (unsigned)__double2loint(v), sg = (unsigned)hi & 0x80000000u;
    const int e = min(((hi >> 20) & 0x7FF) - 896 + k, 254);
    const unsigned m = (((unsigned)hi & 0xFFFFFu) << 3) | (lo >> 29);
    ff_f2 r;
    r.x = (e <= 0) ? 0.0f : __uint_as_float(sg | ((unsigned)e << 23) | m);
    r.y = (e <= 52) ? 0.0f
                    : __uint_as_float(sg | __float_as_uint((float)(lo & 0x1FFFFFFFu) * __uint_as_float((unsigned)(e - 52) << 23)));
    return r;
}

// two-float sum and product (a few 2^-47; ff_f2 parts need not be normalised)
__device__ __forceinline__ ff_f2 ff_add2(const ff_f2 &a, const ff_f2 &b)
{
    float s, e;
    ff_two_sum(a.x, b.x, s, e);
    e = ff_add(e, ff_add(a.y, b.y));
    ff_f2 r;
    ff_fast_sum(s, e, r.x, r.y);
    return r;
}

__device__ __forceinline__ ff_f2 ff_mul2(const ff_f2 &a, const ff_f2 &b)
{
    float p, e;
    ff_two_mul(a.x, b.x, p, e);
    e = ff_fma(a.x, b.y, ff_fma(a.y, b.x, e));
    ff_f2 r;
    ff_fast_sum(p, e, r.x, r.y);
    return r;
}

// v 2^k (v in single precision's normal range or 0; the result a normal number)
__device__ __forceinline__ double ff_up(float v, int k)
{
    const unsigned b = __float_as_uint(v);
    const unsigned ef = (b >> 23) & 0xFFu;
    if (ef == 0) return 0.0;
    return __hiloint2double((int)((b & 0x80000000u) | ((unsigned)((int)ef + 896 + k) << 20) | ((b & 0x7FFFFFu) >> 3)),
                            (int)(b << 29));
}

// doubles compared as integers
__device__ __forceinline__ long long ff_ord(double v)
{
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFll);
}

__device__ __forceinline__ float ff_sqrtf(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Least stopping constant of eq. (4.12) for split sweeps: below it the test asks for
// less than their sums' noise, and a root goes on between neighbouring values until
// its bracket is a few ulps wide.  Sweeps per root, FP64 / split, 100 problems of up to
// 400 poles: 5.14 / 5.19 at 0.1, 5.38 / 6.52 at 0.01, 6.6 / 10.7 at 1e-4 (and the default
// max_iter too few)
constexpr double SPLIT_STOP = 0.1;

struct Root {
    int k, m, K, phase, nsw;
    bool last, plain;
    double dK, y, lo, hi;
    double d0, d1, w0, w1, W;   // d_k, d_{k+1}, w_k, w_{k+1}, sum w

    // plain (ablation of the local shifting): the origin is 0 instead of a
    // pole, so y is the root's position itself and every difference
    // (d_j - dK) - y is d_j - lambda formed from rounded values
    __device__ void init(const double *__restrict__ dk, const double *__restrict__ zk, int k_, int m_, double W_,
                         bool plain_ = false)
    {
        k = k_; m = m_; W = W_; plain = plain_;
        last = (k == m - 1);
        d0 = dk[k];
        double z0 = zk[k];
        w0 = z0 * z0;
        if (!last) { d1 = dk[k + 1]; double z1 = zk[k + 1]; w1 = z1 * z1; }
        else       { d1 = d0; w1 = 0.0; }
        phase = 0; nsw = 0;
        K = k; dK = plain ? 0.0 : d0;
        y = last ? 0.5 * W : 0.5 * (d1 - d0);     // midpoint sweep
        if (plain) y += d0;
        lo = hi = 0.0;
    }

    // returns true when the root is final
    __device__ bool update(const Acc &A, double tol, int max_iter, int32_t *status)
    {
        nsw++;
        double f = 1.0 + A.psi + A.phi;
        if (!isfinite(f)) { sdc_latch(status, SUPERDC_DEV_NONFINITE); return true; }
        if (phase == 0) {
            // origin choice (Section 4.2.1) and initial guess: freeze the
            // non-adjacent terms at the midpoint, solve the two-pole model
            if (!last) {
                double D = d1 - d0, h = 0.5 * D;
                double rest = f + w0 / h - w1 / (D - h);
                if (f >= 0.0) { K = k;     lo = 0.0; hi = h;   dK = d0; }
                else          { K = k + 1; lo = -h;  hi = 0.0; dK = d1; }
                if (plain) { lo += dK; hi += dK; dK = 0.0; }
                double a = d0 - dK, b = d1 - dK;     // one of them is 0 unless plain
                y = quad_in(rest, -(rest * (a + b) + w0 + w1), w0 * b + w1 * a + rest * a * b, lo, hi);
            } else {
                double ym = 0.5 * W;
                if (f >= 0.0) { lo = 0.0; hi = ym; } else { lo = ym; hi = W; }
                double rest = f + w0 / ym;
                y = (rest > 0.0) ? w0 / rest : 0.5 * (lo + hi);
                if (!(y > lo && y < hi)) y = 0.5 * (lo + hi);
                if (plain) { y += d0; lo += d0; hi += d0; }
            }
            phase = 1;
            return false;
        }
        if (fabs(f) < tol * (1.0 + fabs(A.psi) + fabs(A.phi))) return true;   // eq. (4.12)
        if (f < 0.0) lo = y; else hi = y;
        double ynew;
        if (!last) {
            // middle-way step: psi ~ a1 + b1/(d_k - x), phi ~ a2 + b2/(d_{k+1} - x)
            double Dk = (d0 - dK) - y, Dk1 = (d1 - dK) - y;
            double c = f - Dk * A.dpsi - Dk1 * A.dphi;
            double Aq = (Dk + Dk1) * f - Dk * Dk1 * (A.dpsi + A.dphi);
            double Bq = Dk * Dk1 * f;
            double corr;
            if (c == 0.0) {
                corr = (Aq != 0.0) ? Bq / Aq : 0.0;
            } else {
                double disc = Aq * Aq - 4.0 * Bq * c;
                if (disc < 0.0) disc = 0.0;
                double s = sqrt(disc);
                double den = Aq + (Aq >= 0 ? s : -s);
                corr = (den != 0.0) ? 2.0 * Bq / den : 0.0;
            }
            ynew = y + corr;
        } else {
            double Dl = (d0 - dK) - y;
            double den = f - Dl * A.dpsi;
            double corr = (den != 0.0) ? Dl + Dl * Dl * A.dpsi / den : 0.0;
            ynew = y + corr;
        }
        if (!(ynew > lo && ynew < hi)) ynew = lo + 0.5 * (hi - lo);
        if (ynew == y || !(ynew > lo && ynew < hi)) return true;   // bracket at double resolution
        y = ynew;
        if (nsw - 1 >= max_iter) { sdc_latch(status, SUPERDC_DEV_NOCONV); return true; }
        return false;
    }

    // The same step after a split sweep (not the last root).  S: sums without the
    // two poles next to the root, in units of 2^(kk + kw), the far fields' single
    // precision parts added; low: their FP64 part.  Only what decides the root's
    // accuracy is FP64: the function value (two reciprocals, the adjacent poles'
    // terms, the joined sums) and the new iterate, 18 instructions of 16 cycles of
    // the SM each; update(), with two divisions, a square root, 9 comparisons
    // (two slots each) and the sums it wants in FP64, takes about 88.  The step is
    // two floats where its error stays in the last iterate (the roots that stop
    // are as accurate as after FP64 steps), single precision where it does not
    // (stopping test's scale, middle-way factor, initial guess), in units of the
    // spread; signs and order are integer comparisons.  Values out of single
    // precision's range (a root within 2^-50 of the spread of its pole, tiny
    // weights) go to update().  Measured with the mixed series of the far fields
    // (GB300, 4096 problems of 32..2048 poles): the step 24.6 -> 22.2 ms, one
    // small batch 0.335 -> 0.310; roots' errors and sweep counts unchanged
    // against quadruple precision (single precision steps: median error 4.0e-15
    // -> 5.5e-15).
    __device__ __forceinline__ bool update_split(const FfAcc &S, double low, int kk, int kw, double tol, int max_iter,
                                                 int32_t *status)
    {
        const int kf = kk + kw;
        const bool right = K != k;
        const double D = d1 - d0, ay = fabs(y), g = D - ay;
        const double wn = right ? w1 : w0, wf = right ? w0 : w1;
        const double rn = rcp_nr2(ay), rf = rcp_nr2(g);
        const double c1 = ff_pow2(kf);
        const double rest = fma((double)S.s, c1, fma((double)S.sl, c1, 1.0 + low));
        const double u = fma(wf, rf, -(wn * rn));
        const double f = rest + (right ? -u : u);
        const int ef = fexp(f), er = fexp(rest);
        const bool fit = abs(kf) < 50 && fexp(ay) + kk > 973 && fexp(wn) - kw > 923 && fexp(wf) - kw > 923 &&
                         ef - kf < 1073 && er - kf < 1073;
        if (!fit) {
            // a gap at the end of the exponent range (a weight whose square is subnormal)
            // has no reciprocal: the guess stands
            if (phase != 0 && fexp(ay) < 31) return true;
            const double c2 = ff_pow2(kf + kk), an = wn * rn, af = wf * rf;
            Acc A;
            A.psi = fma((double)S.psi, c1, right ? -af : -an);
            A.phi = (f - 1.0) - A.psi;
            A.dpsi = fma((double)S.dpsi, c2, right ? af * rf : an * rn);
            A.dphi = fma((double)S.dphi, c2, right ? an * rn : af * rf);
            return update(A, tol, max_iter, status);
        }
        nsw++;
        if (phase == 0) {
            // origin choice and initial guess: see update(); y = -v right of the middle
            const float Wn = ff_top(wn, -kw), Wf = ff_top(wf, -kw);
            const float Df = ff_top(D, kk), R = ff_top(rest, -kf), h = 0.5f * Df;
            const bool rt = __double2hiint(f) < 0;
            const float W2 = Wn + Wf;
            const float qb = -fmaf(R, Df, rt ? -W2 : W2), qc = (rt ? -Wf : Wn) * Df;
            const float disc = fmaf(qb, qb, -4.0f * R * qc);
            const float q = -0.5f * (qb + copysignf(ff_sqrtf(fmaxf(disc, 0.0f)), qb));
            const float v1 = q * mufu_rcp(R), v2 = qc * mufu_rcp(q);    // a guess: approximations do
            float v = 0.5f * h;
            if (disc >= 0.0f) {
                if (v1 > 0.0f && v1 < h) v = v1;
                else if (v2 > 0.0f && v2 < h) v = v2;
            }
            const double hd = 0.5 * D;
            K = rt ? k + 1 : k;
            dK = rt ? d1 : d0;
            lo = rt ? -hd : 0.0;
            hi = rt ? 0.0 : hd;
            y = ff_up(rt ? -v : v, -kk);
            phase = 1;
            return false;
        }
        const float one = __int_as_float((127 - kf) << 23);
        const ff_f2 F = ff_split2(f, -kf), N2 = ff_split2(ay, kk), G2 = ff_split2(g, kk);
        ff_f2 an, af, bn, bf;                     // w / t and w / t^2 of the two poles
        ff_div(ff_split2(wn, -kw), N2.x, N2.y, an.x, an.y);
        ff_div(ff_split2(wf, -kw), G2.x, G2.y, af.x, af.y);
        const float psi = S.psi - (right ? af.x : an.x), phi = (F.x - one) - psi;
        if (fabsf(F.x) < (float)tol * (one + fabsf(psi) + fabsf(phi))) return true;   // eq. (4.12)
        if (__double2hiint(f) < 0) lo = y; else hi = y;
        ff_div(an, N2.x, N2.y, bn.x, bn.y);
        ff_div(af, G2.x, G2.y, bf.x, bf.y);
        const float dpsi = S.dpsi + (right ? bf.x : bn.x), dphi = S.dphi + (right ? bn.x : bf.x);
        const ff_f2 p = right ? G2 : N2, q = right ? N2 : G2;
        // middle-way step 2 B / (A +- sqrt(A^2 - 4 B C)), A = (q - p) f + p q f', B = -p q f,
        // C = f + p psi' - q phi': t (1 + e), t = B / A, e = h / (1 + sqrt(1 - h))^2, h = 4 t C / A
        const ff_f2 pq = ff_mul2(p, q);
        const ff_f2 A = ff_add2(ff_mul2(ff_add2(q, ff_f2{-p.x, -p.y}), F),
                                ff_mul2(pq, ff_add2(ff_add2(bn, bf), ff_f2{S.dpsi + S.dphi, 0.0f})));
        const ff_f2 nb = ff_mul2(pq, F);
        float t, tl;
        ff_div(ff_f2{-nb.x, -nb.y}, A.x, A.y, t, tl);
        const float hh = 4.0f * t * (fmaf(p.x, dpsi, fmaf(-q.x, dphi, F.x)) * mufu_rcp(A.x));
        const float r1 = mufu_rcp(1.0f + ff_sqrtf(fmaxf(1.0f - hh, 0.0f)));
        const float corr = t, corl = fmaf(t, hh < 1.0f ? hh * r1 * r1 : 1.0f, tl);
        const long long ol = ff_ord(lo), oh = ff_ord(hi);
        double yn = y;
        bool in = fabsf(corr) < 2.0f && fabsf(corl) < 2.0f;      // also not NaN
        if (in) {
            yn = (y + ff_up(corl, -kk)) + ff_up(corr, -kk);
            const long long on = ff_ord(yn);
            in = on > ol && on < oh;
        }
        if (!in) {
            yn = lo + 0.5 * (hi - lo);
            const long long on = ff_ord(yn);
            in = on > ol && on < oh;
        }
        if (!in || __double_as_longlong(yn) == __double_as_longlong(y)) return true;  // bracket at double resolution
        y = yn;
        if (nsw - 1 >= max_iter) { sdc_latch(status, SUPERDC_DEV_NOCONV); return true; }
        return false;
    }
};

// The last root of a problem (right of every pole), by one warp: the lanes
// split the poles, every lane holds the same iterate.
__device__ __forceinline__ void last_root_warp(const double *__restrict__ dk, const double *__restrict__ zk, int m,
                                               double W, double tol, int max_iter, int32_t *status, Root &R)
{
    const int lane = threadIdx.x & 31;
    R.init(dk, zk, m - 1, m, W);
    for (bool fin = false; !fin;) {
        Acc A = {0.0, 0.0, 0.0, 0.0};
        for (int j = lane; j < m; j += 32) {
            const double r = rcp_nr1(shifted_t(dk[j], R.dK, R.y));
            const double z = zk[j];
            const double a = (z * z) * r;
            A.psi += a;
            A.dpsi = fma(a, r, A.dpsi);
        }
        for (int sh = 16; sh > 0; sh >>= 1) {
            A.psi += __shfl_xor_sync(0xffffffffu, A.psi, sh);
            A.dpsi += __shfl_xor_sync(0xffffffffu, A.dpsi, sh);
        }
        fin = R.update(A, tol, max_iter, lane == 0 ? status : nullptr);
    }
}

// p 2^ex *= f, p kept in [1/2, 1) (zero, subnormal and non-finite products pass through)
__device__ __forceinline__ void exp_mul(double &p, int &ex, double f)
{
    p *= f;
    const int h = __double2hiint(p), e = (h >> 20) & 0x7FF;
    if (e != 0 && e != 0x7FF) {
        ex += e - 1022;
        p = __hiloint2double((h & 0x800FFFFF) | (1022 << 20), __double2loint(p));
    }
}

// The factors of zhat_i that the integer products leave out: the eigenvalues
// next to d_i (j = i - 1, i) with their poles, and the last one (j = m - 1).
// pn / pd 2^ex is multiplied by them.
__device__ __forceinline__ void lowner_edges(const double *__restrict__ dk, const double *__restrict__ dorg,
                                             const double *__restrict__ eta, double di, int i, int m, double &pn,
                                             double &pd, int &ex)
{
    int xd = 0;
    exp_mul(pn, ex, (dorg[m - 1] - di) + eta[m - 1]);
    if (i < m - 1) {
        exp_mul(pn, ex, (dorg[i] - di) + eta[i]);
        exp_mul(pd, xd, dk[m - 1] - di);
    }
    if (i > 0) {
        exp_mul(pn, ex, (dorg[i - 1] - di) + eta[i - 1]);
        exp_mul(pd, xd, dk[i - 1] - di);
    }
    ex -= xd;
}

}  // namespace
