// qlga_fixed.cuh -- the FP64 potential unitary in 64-bit integer fixed point.
//
// GB300 issues one FP64 instruction per SM sub-partition every 64-76 cycles (measured: DFMA 64, DADD and
// DMUL 76, FP64 <-> FP32 conversions 64) but a 32 x 32 + 64-bit integer multiply-add every 4.4, a
// 64-bit addition every 2.4 and an FP32 multiply-add every cycle.  A product of two fixed-point numbers
// takes three of the first, so U on a site costs a quarter of its FP64 form, at a finer
// resolution: relative to the site's largest component the operands carry 2^-58, where FP64 rounds
// every operation at 2^-53 of its own result.
//
// Numbers.  A site's psi = a + b and d = a - b are int64 with one exponent per vector, psi's largest
// component in [2^57, 2^58).  An operand of a product is split as v = h 2^32 + l, l the low word
// taken as signed; h h' and h l' + l h' are summed in 64-bit accumulators, and l l' (zero mean,
// below 2^62) is dropped but in the squares of the density.  The entries of delta W and the phase are fixed point with
// 2^61 = 1.  (Cross terms in FP32 are 13% of a 1024^2 step, 5.65 against 6.54 ms for ten with load and read-out, but round the
// low limb of an entry to 24 bits: the phase and W's diagonal, which sites of one density share, were
// off by up to 2^-55 whatever their size, 7e-17 a step of a run's phase.)
//
// U = e^{-i delta c} exp(-i delta W) as in potential_site, by the plain Taylor sum: the terms
// T_k = (-i delta W)^k x are formed in fixed point up to the order k0 - 1 whose successor is bounded
// by beta^k0 / k0! <= 2^-31 and added as T_k / k!; the terms from k0 on, so small that FP32 carries
// them to 2^-54 of the site, continue in FP32 to a bound of 2^-57.  The phase is applied as v + (e^{-i delta c} - 1) v.
//
// Domain.  beta <= 0.25 and finite components below 2^60; a warp with a lane outside it (among them
// every site that the status word reports) takes the FP64 code.  Components below 2^-59 of the
// site's largest one, and sites below 2^-850, round to zero.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

namespace qlga {

#define QLGA_HD __host__ __device__ __forceinline__

using i64 = long long;

// ------------------------------------------------------------------ numbers

struct Limb {
    int h, l;  // h 2^32 + l
};

QLGA_HD Limb fx_split(i64 v) {  // the low limb is the low word as it stands, the high one takes its sign
    return {int(v >> 32) + int(unsigned(v) >> 31), int(unsigned(v))};
}

// s + a b, 32 x 32 bits: one instruction
QLGA_HD i64 fx_mad(int a, int b, i64 s) {
#ifdef __CUDA_ARCH__
    i64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(s));
    return d;
#else
    return s + i64(a) * b;
#endif
}

// The running sum of products: hh 2^64 + mid 2^32
struct FxAcc {
    i64 hh, mid;
};
QLGA_HD void fx_mac(FxAcc& s, Limb a, Limb b) {
    s.hh = fx_mad(a.h, b.h, s.hh);
    s.mid = fx_mad(a.l, b.h, fx_mad(a.h, b.l, s.mid));
}
// Every sum is rounded to nearest, not down: half a unit a step would add up over a run's thousands.
template <int N>
QLGA_HD FxAcc fx_zero() { return {0, i64(1) << (N - 33)}; }
QLGA_HD FxAcc operator-(FxAcc a, FxAcc b) { return {a.hh - b.hh, a.mid - b.mid}; }  // a limb of -2^31 has no negative
template <int N>
QLGA_HD i64 fx_sum(FxAcc s) {  // sum / 2^N, 32 < N < 64, of an accumulator that began as fx_zero<N>
    return (s.hh << (64 - N)) + (s.mid >> (N - 32));
}
// a b / 2^N with l l' too, for factors that need not fill their limbs
template <int N>
QLGA_HD i64 fx_mul_full(Limb a, Limb b) {
    FxAcc s = fx_zero<N>();
    fx_mac(s, a, b);
    s.mid += fx_mad(a.l, b.l, 0) >> 32;
    return fx_sum<N>(s);
}
QLGA_HD i64 fx_mul(Limb a, Limb b) {  // a b / 2^61
    FxAcc s = fx_zero<61>();
    fx_mac(s, a, b);
    return fx_sum<61>(s);
}

// v 2^n for n in [-63, 62], rounded to nearest (|v| < 2^62; the caller knows that it fits)
QLGA_HD i64 fx_scale(i64 v, int n) {
    const int nl = n > 0 ? n : 0, nr = n < 0 ? -n : 0;
    return (((v << nl << 1) >> nr) + 1) >> 1;
}

template <class T>
QLGA_HD int fx_clz(T v) {  // v != 0
#ifdef __CUDA_ARCH__
    return __clzll(v);
#else
    return __builtin_clzll(static_cast<unsigned long long>(v));
#endif
}

// ------------------------------------------------------------------ constants

// float of a fixed-point value times the float c
QLGA_HD float fx_float(Limb v, float c) { return fmaf(float(v.h), 4294967296.f * c, float(v.l) * c); }
QLGA_HD int fx_rint(float x) {
#ifdef __CUDA_ARCH__
    return __float2int_rn(x);
#else
    return int(rintf(x));
#endif
}

// A coupling c = m 2^(ex - 60), m in [2^59, 2^60) (0: all zero)
struct FxConst {
    Limb m;
    int ex;
    FxConst() = default;
    __host__ explicit FxConst(double c) : m{0, 0}, ex(0) {
        if (c == 0.0) return;
        int e;
        const double f = std::frexp(c, &e);  // c = f 2^e, |f| in [1/2, 1)
        m = fx_split(i64(std::ldexp(f, 60)));
        ex = e;
    }
};

// The potential's constants (those of PotConst, qlga_device.cuh) for the fixed-point form.
struct FixPot {
    FxConst cphase, dz, dr, e0, R;
    float b1, b2, cphase_f, R_f;
    FixPot() = default;
    __host__ FixPot(double cphase_, double dz_, double dr_, double e0_, double R_, double b1_, double b2_)
        : cphase(cphase_), dz(dz_), dr(dr_), e0(e0_), R(R_), b1(float(b1_)), b2(float(b2_)), cphase_f(float(cphase_)),
          R_f(float(R_)) {}
};

struct FxCpxF {
    float re, im;
};

// num / den in 2^61 = 1
QLGA_HD constexpr i64 fx_ratio(i64 num, i64 den) { return ((num << 61) + den / 2) / den; }
constexpr i64 kFxR32m1 = 518226390554926330LL;  // sqrt(3/2) - 1 in 2^61 = 1

// 1/k! in 2^61 = 1, k = 0..kFxTerms
constexpr int kFxTerms = 16;
struct FxInvFact {
    int h[kFxTerms + 1], l[kFxTerms + 1];
};
constexpr FxInvFact make_fx_inv_fact() {
    FxInvFact t{};
    i64 f = 1;
    for (int k = 0; k <= kFxTerms; ++k) {
        if (k) f *= k;
        const i64 v = fx_ratio(1, f), h = (v + (i64(1) << 31)) >> 32;
        t.h[k] = int(h);
        t.l[k] = int(v - h * (i64(1) << 32));
    }
    return t;
}
static constexpr FxInvFact kFxInvFactHost = make_fx_inv_fact();
__constant__ FxInvFact c_fx_inv_fact = make_fx_inv_fact();
QLGA_HD Limb fx_inv_fact(int k) {
#ifdef __CUDA_ARCH__
    return {c_fx_inv_fact.h[k], c_fx_inv_fact.l[k]};
#else
    return {kFxInvFactHost.h[k], kFxInvFactHost.l[k]};
#endif
}

// ------------------------------------------------------------------ double <-> fixed point

QLGA_HD unsigned fx_hi(double x) {
#ifdef __CUDA_ARCH__
    return unsigned(__double2hiint(x));
#else
    unsigned long long u;
    std::memcpy(&u, &x, 8);
    return unsigned(u >> 32);
#endif
}
QLGA_HD unsigned fx_lo(double x) {
#ifdef __CUDA_ARCH__
    return unsigned(__double2loint(x));
#else
    unsigned long long u;
    std::memcpy(&u, &x, 8);
    return unsigned(u);
#endif
}
QLGA_HD unsigned fx_top(unsigned m, double x) {  // the larger of m and x's high word without sign
    const unsigned h = fx_hi(x) & 0x7fffffffu;
    return h > m ? h : m;
}
QLGA_HD double fx_bits(unsigned hi, unsigned lo) {
#ifdef __CUDA_ARCH__
    return __hiloint2double(int(hi), int(lo));
#else
    const unsigned long long u = (static_cast<unsigned long long>(hi) << 32) | lo;
    double x;
    std::memcpy(&x, &u, 8);
    return x;
#endif
}
QLGA_HD double fx_pow2(int e) { return fx_bits(unsigned(e + 1023) << 20, 0u); }  // 2^e, -1022 <= e <= 1023

// The biased exponent that a set of doubles is converted with: m is the largest high word without
// sign; every |x| < 2^(E - 1022).  kFxMinExp: smaller sets round to zero.
constexpr int kFxMinExp = 1022 - 850;
QLGA_HD int fx_exponent(unsigned m) {
    const int e = int(m >> 20);
    return e > kFxMinExp ? e : kFxMinExp;
}

// x 2^(BITS + 1022 - E), rounded to nearest: the fixed-point value, below 2^BITS, of a double of a set
// with exponent E
template <int BITS>
QLGA_HD i64 fx_from_double(double x, int E) {
    const unsigned hi = fx_hi(x), lo = fx_lo(x);
    int dE = E - int((hi >> 20) & 0x7ffu);
    dE = dE < 63 ? dE : 63;
    const unsigned long long M = (static_cast<unsigned long long>((hi & 0xfffffu) | 0x100000u) << 32) | lo;
    const i64 v = (i64((M << (BITS - 52)) >> dE) + 1) >> 1;
    const i64 s = i64(int(hi)) >> 63;
    return (v ^ s) - s;
}

// v 2^e, rounded to nearest, on integers: where the FP64 pair of FxToDouble would be on a warp's
// critical path.  The result is a normal number (e >= -1022) or zero.
QLGA_HD double fx_pack(i64 v, int e) {
    unsigned long long m = static_cast<unsigned long long>(v < 0 ? -v : v);
    if (m == 0) return 0.0;
    const int lz = fx_clz(m);
    m <<= lz;
    const unsigned long long r = (m >> 11) + ((m >> 10) & 1);  // [2^52, 2^53]: its top bit counts one exponent
    const unsigned long long u = (static_cast<unsigned long long>(e + 63 - lz + 1022) << 52) + r;
    return fx_bits(unsigned(u >> 32) | (unsigned(v >> 63) & 0x80000000u), unsigned(u));
}

// v 2^e (|v| < 2^62, -1022 <= e): one rounding.  scale_hi = 2^(e + 32), scale_lo = 2^e,
// off = -(2^52 + 2^31) 2^(e + 32) - 2^(e + 52).  Two FP64 instructions: they run beside the integer work.
struct FxToDouble {
    double hi, lo, off;
    QLGA_HD explicit FxToDouble(int e) : hi(fx_pow2(e + 32)), lo(fx_pow2(e)) {
        // 2^(e + 84) + 2^(e + 63) + 2^(e + 52): 33 bits
        off = -fx_bits((unsigned(e + 84 + 1023) << 20), 0x80000000u + 0x00100000u) ;
    }
    QLGA_HD double operator()(i64 v) const {
        const double dh = fx_bits(0x43300000u, unsigned(int(v >> 32)) ^ 0x80000000u);  // 2^52 + 2^31 + high word
        const double dl = fx_bits(0x43300000u, unsigned(v));                           // 2^52 + low word
        return fma(dl, lo, fma(dh, hi, off));
    }
};

// ------------------------------------------------------------------ the site

struct FxVec {
    Limb re[5], im[5];
};

// Shift that brings the largest of the ten components of (re, im) to [2^57, 2^58): v -> v 2^(-n).
// Returns n (components below 2^62; all zero: -57).
QLGA_HD int fx_headroom(const i64 re[5], const i64 im[5]) {
    unsigned long long m = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) m |= static_cast<unsigned long long>(re[i] ^ (re[i] >> 63)) | static_cast<unsigned long long>(im[i] ^ (im[i] >> 63));
    return m ? 6 - fx_clz(m) : -57;  // 64 - clz bits now, 58 wanted
}
QLGA_HD i64 fx_shift(i64 v, int n) { return fx_scale(v, -n); }  // v 2^(-n), n in [-57, 5] (|v| < 2^(58 + n) and 2^62)

// delta W of a site in fixed point (2^61 = 1)
struct FxW {
    Limb D[5];
    Limb e0r, e0i, e1r, e1i;  // delta g1 F_+ times 1 and sqrt(3/2)
    FxVec u;                  // u_j = (-1)^j psi_{4-j}
    Limb R;                   // delta g2 / 5: G = R dot / 2^55
    float Rf;
};

// t <- -i delta W t
QLGA_HD void fx_apply(const FxW& W, const FxVec& t, i64 ore[5], i64 oim[5]) {
    FxAcc tp = fx_zero<60>(), tn = {0, 0}, ti = fx_zero<60>();
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        fx_mac(tp, W.u.re[j], t.re[j]);
        fx_mac(tn, W.u.im[j], t.im[j]);
        fx_mac(ti, W.u.re[j], t.im[j]);
        fx_mac(ti, W.u.im[j], t.re[j]);
    }
    const Limb Gr = fx_split(fx_mul_full<55>(W.R, fx_split(fx_sum<60>(tp - tn))));
    const Limb Gi = fx_split(fx_mul_full<55>(W.R, fx_split(fx_sum<60>(ti))));
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        // y = (W t)_i; o = -i y: o.re = y.im, o.im = -y.re
        FxAcc yr = fx_zero<61>(), yi = fx_zero<61>(), nr = {0, 0}, ni = {0, 0};
        fx_mac(yr, W.D[i], t.re[i]);
        fx_mac(yi, W.D[i], t.im[i]);
        fx_mac(yr, W.u.re[i], Gr);  // conj(u) G
        fx_mac(yr, W.u.im[i], Gi);
        fx_mac(yi, W.u.re[i], Gi);
        fx_mac(ni, W.u.im[i], Gr);
        if (i > 0) {  // e t_{i-1}
            const bool s = i == 1 || i == 4;
            const Limb er = s ? W.e0r : W.e1r, ei = s ? W.e0i : W.e1i;
            fx_mac(yr, er, t.re[i - 1]);
            fx_mac(nr, ei, t.im[i - 1]);
            fx_mac(yi, er, t.im[i - 1]);
            fx_mac(yi, ei, t.re[i - 1]);
        }
        if (i < 4) {  // conj(e) t_{i+1}
            const bool s = i == 0 || i == 3;
            const Limb er = s ? W.e0r : W.e1r, ei = s ? W.e0i : W.e1i;
            fx_mac(yr, er, t.re[i + 1]);
            fx_mac(yr, ei, t.im[i + 1]);
            fx_mac(yi, er, t.im[i + 1]);
            fx_mac(ni, ei, t.re[i + 1]);
        }
        ore[i] = fx_sum<61>(yi - ni);
        oim[i] = -fx_sum<61>(yr - nr);
    }
}

// 1/k, k = 1..kFxDegree, without a division
constexpr int kFxDegree = 24;
struct FxInv {
    float v[kFxDegree + 1];
};
constexpr FxInv make_fx_inv() {
    FxInv t{};
    for (int k = 1; k <= kFxDegree; ++k) t.v[k] = float(1.0 / k);
    return t;
}
static constexpr FxInv kFxInvHost = make_fx_inv();
__constant__ FxInv c_fx_inv = make_fx_inv();
QLGA_HD float fx_inv(int k) {
#ifdef __CUDA_ARCH__
    return c_fx_inv.v[k];
#else
    return kFxInvHost.v[k];
#endif
}

constexpr float kFxBetaMax = 0.25f;
// Truncation of the Taylor sums, relative to the site: the same terms are missing from step to step, so
// the bound is a sixteenth of FP64's 2^-53 (a term of the FP32 part costs 2% of U).  Orders whose bound is
// above kFxTolF run in fixed point.
constexpr float kFxTol = 6.9388939e-18f;   // 2^-57
constexpr float kFxTolF = 4.6566129e-10f;  // 2^-31

// Smallest K with beta^(K+1)/(K+1)! <= tol (beta <= 1: at most 19 for 2^-57)
QLGA_HD int fx_degree(float beta, float tol) {
    int K = 0;
    float term = beta;
    while (term > tol && K < kFxDegree - 1) {
        ++K;
        term *= beta * fx_inv(K + 1);
    }
    return K;
}

// t <- (-i / k) delta W t in FP32
QLGA_HD void fx_apply_f(const FxW& W, const FxCpxF u[5], const FxCpxF t[5], FxCpxF o[5], float ik) {
    float ar = 0.f, ai = 0.f;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        ar = fmaf(u[j].re, t[j].re, fmaf(-u[j].im, t[j].im, ar));
        ai = fmaf(u[j].re, t[j].im, fmaf(u[j].im, t[j].re, ai));
    }
    const float gr = W.Rf * ar, gi = W.Rf * ai;
    const float s61 = 4.3368087e-19f;  // 2^-61
    const float e0rf = fx_float(W.e0r, s61), e0if = fx_float(W.e0i, s61);
    const float e1rf = fx_float(W.e1r, s61), e1if = fx_float(W.e1i, s61);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const float Df = fx_float(W.D[i], s61);
        float yr = fmaf(Df, t[i].re, fmaf(u[i].re, gr, u[i].im * gi));
        float yi = fmaf(Df, t[i].im, fmaf(u[i].re, gi, -u[i].im * gr));
        if (i > 0) {
            const bool s = i == 1 || i == 4;
            const float er = s ? e0rf : e1rf, ei = s ? e0if : e1if;
            yr = fmaf(er, t[i - 1].re, fmaf(-ei, t[i - 1].im, yr));
            yi = fmaf(er, t[i - 1].im, fmaf(ei, t[i - 1].re, yi));
        }
        if (i < 4) {
            const bool s = i == 0 || i == 3;
            const float er = s ? e0rf : e1rf, ei = s ? e0if : e1if;
            yr = fmaf(er, t[i + 1].re, fmaf(ei, t[i + 1].im, yr));
            yi = fmaf(er, t[i + 1].im, fmaf(-ei, t[i + 1].re, yi));
        }
        o[i] = {ik * yi, -ik * yr};
    }
}

// The quadratic forms of psi (unit 2^(2 e + 60) for components of unit 2^e)
struct FxForms {
    i64 rho, Fz, Fpr, Fpi;  // F_+ = 2 (Fpr + i Fpi)
};

QLGA_HD void fx_forms(const FxVec& p, FxForms& f) {
    const Limb *re = p.re, *im = p.im;
    i64 n[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {  // with l l': of a square it has no zero mean
        FxAcc s = fx_zero<60>();
        fx_mac(s, re[i], re[i]);
        fx_mac(s, im[i], im[i]);
        s.mid += (fx_mad(re[i].l, re[i].l, 0) >> 32) + (fx_mad(im[i].l, im[i].l, 0) >> 32);
        n[i] = fx_sum<60>(s);
    }
    f.rho = (n[0] + n[1]) + (n[2] + n[3]) + n[4];
    f.Fz = 2 * (n[0] - n[4]) + (n[1] - n[3]);
    i64 fr[2], fi[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {  // conj(p0) p1 + conj(p3) p4, then conj(p1) p2 + conj(p2) p3
        const int a = q, b = q == 0 ? 3 : 2;
        FxAcc r = fx_zero<60>(), i = fx_zero<60>(), n = {0, 0};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int j = k ? b : a;
            fx_mac(r, re[j], re[j + 1]);
            fx_mac(r, im[j], im[j + 1]);
            fx_mac(i, re[j], im[j + 1]);
            fx_mac(n, im[j], re[j + 1]);
        }
        fr[q] = fx_sum<60>(r);
        fi[q] = fx_sum<60>(i - n);
    }
    const Limb r = fx_split(kFxR32m1);
    f.Fpr = fr[0] + fr[1] + fx_mul(r, fx_split(fr[1]));
    f.Fpi = fi[0] + fi[1] + fx_mul(r, fx_split(fi[1]));
}

QLGA_HD float fx_pow2f(int n) {  // 2^n, clamped to the normal range
    n = n < -126 ? -126 : (n > 127 ? 127 : n);
    union {
        unsigned u;
        float f;
    } p;
    p.u = unsigned(n + 127) << 23;
    return p.f;
}

// e^{-i theta} - 1 = (-c, -s), theta and the results in 2^61 = 1, |theta| <= 1/4: the Taylor series of
// sin and cos, the terms that FP32 carries to 2^-57 evaluated in it.
QLGA_HD void fx_phase(i64 theta, i64& c, i64& s) {
    const Limb t = fx_split(theta);
    const Limb q = fx_split(fx_mul(t, t));
    const float qf = fx_float(q, 4.3368087e-19f);  // 2^-61
    const i64 s3 = fx_ratio(1, 5040) - (i64(int(9007199254740992.f * qf * (2.7557319e-6f - qf * 2.5052108e-8f))) << 8);
    const i64 s2 = fx_ratio(1, 120) - fx_mul(q, fx_split(s3));
    const i64 s1 = fx_ratio(1, 6) - fx_mul(q, fx_split(s2));
    s = theta - fx_mul(t, fx_split(fx_mul(q, fx_split(s1))));
    const i64 c3 = fx_ratio(1, 720) - (i64(int(1125899906842624.f * qf * (2.4801587e-5f - qf * (2.7557319e-7f - qf * 2.0876757e-9f)))) << 11);
    const i64 c2 = fx_ratio(1, 24) - fx_mul(q, fx_split(c3));
    const i64 c1 = (i64(1) << 60) - fx_mul(q, fx_split(c2));
    c = fx_mul(q, fx_split(c1));
}

// What the warp decides from: beta and theta of a lane (as upper bounds)
struct FxBounds {
    float beta, theta;
};
QLGA_HD FxBounds fx_bounds(const FxForms& f, int e, const FixPot& C) {
    // the forms in 2^61 = 1, times 2^(2 e + 121)
    const float c = 4.3368087e-19f;
    const float rho = fx_float(fx_split(f.rho), c), fz = fx_float(fx_split(f.Fz), c);
    const float fr = 2.f * fx_float(fx_split(f.Fpr), c), fi = 2.f * fx_float(fx_split(f.Fpi), c);
    const float F = sqrtf(fmaf(fz, fz, fmaf(fr, fr, fi * fi)));
    const float u = 1.00001f * fx_pow2f(2 * e + 121);
    FxBounds b;
    b.beta = u * fmaf(C.b1, F, C.b2 * rho);
    b.theta = u * fabsf(C.cphase_f) * rho;
    return b;
}

// c q 2^(2 e + 60) in 2^61 = 1, twice that for more = 1 (below 2^62)
QLGA_HD i64 fx_coupled(const FxConst& c, i64 q, int e, int more) {
    FxAcc s = fx_zero<60>();
    fx_mac(s, c.m, fx_split(q));
    int n = c.ex + 2 * e + 121 + more;
    n = n < -63 ? -63 : (n > 30 ? 30 : n);
    return fx_scale(fx_sum<60>(s), n);
}

QLGA_HD void fx_singlet(const FixPot& C, int e, Limb& R, float& Rf) {
    // R 2^(2 e) = m 2^(ex - 60 + 2 e); G conj(u) / 2^61 = R 2^(2 e) dot 2^60 conj(u) and G = W.R dot / 2^55.
    // |psi|^2 >= 2^114 and beta <= 0.25 bound W.R by 2^62
    int n = C.R.ex + 2 * e + 116;
    n = n < -63 ? -63 : (n > 30 ? 30 : n);
    R = fx_split(fx_scale((i64(C.R.m.h) * (i64(1) << 32)) + C.R.m.l, n));
    Rf = C.R_f * fx_pow2f(2 * e + 116);  // for u in 2^58 = 1
}

QLGA_HD void fx_build_w(const FxVec& p, const FxForms& f, int e, const FixPot& C, FxW& W) {
    const i64 gz = fx_coupled(C.dz, f.Fz, e, 0), g2r = fx_coupled(C.dr, f.rho, e, 0);
#pragma unroll
    for (int i = 0; i < 5; ++i) W.D[i] = fx_split((2 - i) * gz - g2r);
    const Limb r = fx_split(kFxR32m1);
    const i64 er = fx_coupled(C.e0, f.Fpr, e, 1), ei = fx_coupled(C.e0, f.Fpi, e, 1);
    W.e0r = fx_split(er);
    W.e0i = fx_split(ei);
    W.e1r = fx_split(er + fx_mul(r, fx_split(er)));
    W.e1i = fx_split(ei + fx_mul(r, fx_split(ei)));
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        auto turned = [&](Limb v) { return (j & 1) ? fx_split(-(v.h * (i64(1) << 32) + v.l)) : v; };
        W.u.re[j] = turned(p.re[4 - j]);
        W.u.im[j] = turned(p.im[4 - j]);
    }
    fx_singlet(C, e, W.R, W.Rf);
}

// x <- exp(-i delta W) x for one vector: orders 1..kA in fixed point, kA + 1..K in FP32
QLGA_HD void fx_taylor(const FxW& W, i64 re[5], i64 im[5], int kA, int K) {
    FxVec t;
    i64 tr[5], ti[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        tr[i] = re[i];
        ti[i] = im[i];
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        t.re[i] = fx_split(tr[i]);
        t.im[i] = fx_split(ti[i]);
    }
#pragma unroll 1
    for (int k = 1; k <= kA; ++k) {
        fx_apply(W, t, tr, ti);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            t.re[i] = fx_split(tr[i]);
            t.im[i] = fx_split(ti[i]);
        }
        if (k <= 2) {
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                re[i] += k == 1 ? tr[i] : (tr[i] + 1) >> 1;
                im[i] += k == 1 ? ti[i] : (ti[i] + 1) >> 1;
            }
        } else {
            const Limb f = fx_inv_fact(k);
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                re[i] += fx_mul(f, t.re[i]);
                im[i] += fx_mul(f, t.im[i]);
            }
        }
    }
    if (K > kA) {
        FxCpxF tf[5], sf[5], uf[5], of[5];
        const float s58 = 3.4694470e-18f;  // 2^-58
        const float fact = s58 * fx_float(fx_inv_fact(kA), 4.3368087e-19f);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            tf[i] = {fx_float(t.re[i], fact), fx_float(t.im[i], fact)};
            uf[i] = {fx_float(W.u.re[i], s58), fx_float(W.u.im[i], s58)};
            sf[i] = {0.f, 0.f};
        }
#pragma unroll 1
        for (int k = kA + 1; k <= K; ++k) {
            fx_apply_f(W, uf, tf, of, fx_inv(k));
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                tf[i] = of[i];
                sf[i] = {sf[i].re + of[i].re, sf[i].im + of[i].im};
            }
        }
        const float one = 288230376151711744.f;  // 2^58
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            re[i] += fx_rint(sf[i].re * one);
            im[i] += fx_rint(sf[i].im * one);
        }
    }
}

// x <- x + (e^{-i theta} - 1) x
template <int N = 5>
QLGA_HD void fx_rotate(i64 c, i64 s, i64* re, i64* im) {
    const Limb nc = fx_split(-c), sp = fx_split(s), sn = fx_split(-s);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const Limb r = fx_split(re[i]), m = fx_split(im[i]);
        FxAcc a = fx_zero<61>(), b = fx_zero<61>();
        fx_mac(a, nc, r);
        fx_mac(a, sp, m);
        fx_mac(b, nc, m);
        fx_mac(b, sn, r);
        re[i] += fx_sum<61>(a);
        im[i] += fx_sum<61>(b);
    }
}

// Decisions of a warp; on the host every site is a warp of its own
QLGA_HD bool fx_warp_all(bool v) {
#ifdef __CUDA_ARCH__
    return __all_sync(0xffffffffu, v);
#else
    return v;
#endif
}
QLGA_HD float fx_warp_max(float v) {  // v >= 0
#ifdef __CUDA_ARCH__
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
#else
    return v;
#endif
}

// e^{-i theta} - 1 = (-c, -s) for a theta of any size (fields denser than |theta| = 1/4 are rare)
static __host__ __device__ __noinline__ void fx_phase_large(double theta, i64* c, i64* s) {
    double sn, cs;
    sincos(theta, &sn, &cs);
    *c = i64(rint((1.0 - cs) * 2305843009213693952.0));
    *s = i64(rint(sn * 2305843009213693952.0));
}

// e^{-i theta} - 1 = (-c, -s) of a site from its density, for a warp with a lane beyond |theta| = 1/4 in FP64
QLGA_HD void fx_site_phase(i64 rho, int et, float theta, const FixPot& C, i64& c, i64& s) {
    if (!fx_warp_all(theta <= 0.25f)) {
        const int n = 2 * et < -900 ? -900 : 2 * et;
        const double th = ldexp(double(C.cphase.m.h) * 4294967296.0 + double(C.cphase.m.l), C.cphase.ex + n) * double(rho);
        fx_phase_large(th, &c, &s);
    } else {
        fx_phase(fx_coupled(C.cphase, rho, et, 0), c, s);
    }
}

// U on one site of a warp.  In: psi and d as integers below 2^62 of unit 2^e, `true` amplitudes
// 2^in_log2 times that; ok = false: a lane whose input has no such form.  Out: (psi', d') =
// (U psi, U d) as integers of the unit 2^(returned exponent), below 2^60.  Returns false, with
// nothing changed, if a lane of the warp lies outside the domain.  All 32 lanes take part: the
// orders of the Taylor sums are those of the warp's largest beta.
QLGA_HD bool fx_unitary(i64 pr[5], i64 pi[5], i64 dr[5], i64 di[5], int& e, int in_log2, bool ok,
                                           const FixPot& C) {
    const int np = fx_headroom(pr, pi), nd0 = fx_headroom(dr, di);
    // d goes with psi's unit or, where it is larger, its own, below 2^57 there, so that G of its sums
    // stays below 2^62; psi's sum takes the same unit (its limbs in W have psi's own)
    const int nd = nd0 + 1 > np ? nd0 + 1 : np;
    FxVec p;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        p.re[i] = fx_split(fx_shift(pr[i], np));
        p.im[i] = fx_split(fx_shift(pi[i], np));
    }
    FxForms f;
    fx_forms(p, f);
    const int et = e + np + in_log2;  // exponent of the true psi
    const FxBounds bd = fx_bounds(f, et, C);
    ok = ok && bd.beta <= kFxBetaMax;
    if (!fx_warp_all(ok)) return false;
    const float beta = fx_warp_max(bd.beta);
    const int K = fx_degree(beta, kFxTol), k0 = fx_degree(beta, kFxTolF);
    const int kA = K < k0 ? K : k0;
    FxW W;
    fx_build_w(p, f, et, C, W);
    i64 pc, ps;
    fx_site_phase(f.rho, et, bd.theta, C, pc, ps);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        pr[i] = fx_shift(pr[i], nd);
        pi[i] = fx_shift(pi[i], nd);
        dr[i] = fx_shift(dr[i], nd);
        di[i] = fx_shift(di[i], nd);
    }
#pragma unroll 1
    for (int v = 0; v < 2; ++v) {  // one copy of the code for both vectors
        fx_taylor(W, pr, pi, kA, K);
        fx_rotate(pc, ps, pr, pi);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const i64 tr = pr[i], ti = pi[i];
            pr[i] = dr[i];
            pi[i] = di[i];
            dr[i] = tr;
            di[i] = ti;
        }
    }
    e += nd;
    return true;
}

// U on the pair (a, b) of one site of a warp in FP64, by fx_unitary; the arguments are those of
// potential_site, with in_log2 = -log2 sigma and out_log2 = log2 out_scale.  PQ: (a, b) become
// (P, Q) = (a + i b, a - i b) of the result, summed before the conversion.  Returns false, with nothing changed, outside the domain.
template <bool PQ>
QLGA_HD bool fx_potential(double ar[5], double ai[5], double br[5], double bi[5], int in_log2,
                                             int out_log2, const FixPot& C) {
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        m = fx_top(fx_top(m, ar[i]), ai[i]);
        m = fx_top(fx_top(m, br[i]), bi[i]);
    }
    const bool ok = m < (unsigned(1023 + 60) << 20);  // finite, below 2^60
    const int E = fx_exponent(m);
    int e = E - 1022 - 60;
    i64 pr[5], pi[5], dr[5], di[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const i64 a0 = fx_from_double<60>(ar[i], E), a1 = fx_from_double<60>(ai[i], E);
        const i64 b0 = fx_from_double<60>(br[i], E), b1 = fx_from_double<60>(bi[i], E);
        pr[i] = a0 + b0;
        pi[i] = a1 + b1;
        dr[i] = a0 - b0;
        di[i] = a1 - b1;
    }
    if (!fx_unitary(pr, pi, dr, di, e, in_log2, ok, C)) return false;
    const FxToDouble to(e + out_log2);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const i64 a0 = pr[i] + dr[i], a1 = pi[i] + di[i], b0 = pr[i] - dr[i], b1 = pi[i] - di[i];
        ar[i] = to(PQ ? a0 - b1 : a0);
        ai[i] = to(PQ ? a1 + b0 : a1);
        br[i] = to(PQ ? a0 + b1 : b0);
        bi[i] = to(PQ ? a1 - b0 : b1);
    }
    return true;
}

}  // namespace qlga
