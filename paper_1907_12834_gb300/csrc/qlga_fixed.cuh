// qlga_fixed.cuh -- the FP64 potential unitary in 64-bit integer fixed point.
//
// GB300 issues one FP64 instruction per SM sub-partition every 64-76 cycles (measured: DFMA 64, DADD and
// DMUL 76, FP64 <-> FP32 conversions 64) but a 32 x 32 + 64-bit integer multiply-add every 4.4, a
// 64-bit addition every 2.4 and an FP32 multiply-add every cycle.  A product of two fixed-point numbers
// takes three of the first, so U on a site costs a third of its FP64 form (1024^2 sites of a vortex lattice: 0.60 ms,
// against about 1.7), at a finer resolution: the operands carry 2^-57 of their level, where FP64 rounds
// every operation at 2^-53 of its own result.
//
// Numbers.  Level m of the vectors psi = a + b and d = a - b is a pair of int64 in units of 2^(T_m - 57), with one
// exponent T_m for both vectors: their moduli lie below 2^T_m.  delta W acts between the scaled levels, entry (m, j)
// times 2^(T_j - T_m), in 2^61 = 1; its entries come from psi's own mantissas and exponents, so that no level
// takes its resolution from another (seeds of spin mixing lie many orders of magnitude below the field; with one
// exponent for the site a level at 1e-10 of it kept 1e-7 of its own size).  Where W would add more to a
// level than it holds, T_m is raised to that (fx_budget): FP64, too, rounds the level at what it receives.
// An operand of a product is split as v = h 2^32 + l, l the low word
// taken as signed; h h' and h l' + l h' are summed in 64-bit accumulators, and l l' (zero mean,
// below 2^62) is dropped but in the squares of the density.  (Cross terms in FP32 rounded the low limb of an
// entry to 24 bits: the phase and W's diagonal, which sites of one density share, were
// off by up to 2^-55 whatever their size, 7e-17 a step of a run's phase.)
// The error of a level is 0.36 of 2^-53 (root mean square, of its size and what reaches it), that of the same sum in
// FP64 0.46, from levels of one size to seeds of 1e-40.
//
// U = e^{-i delta c} exp(-i delta W) as in potential_site, by the plain Taylor sum: the terms
// T_k = (-i delta W)^k x are formed in fixed point until the next one is below 2^-31 and added as T_k / k!; the terms from
// there on, so small that FP32 carries them to 2^-54 of the level, continue in FP32 to a bound of 2^-57.  The phase is
// applied as v + (e^{-i delta c} - 1) v.
//
// Domain.  The scaled delta W has a norm of at most 1, components are finite and below 2^60, and a level is empty
// or above 2^-930; a warp with a lane outside it (among them every site that the status word reports) takes the FP64 code.
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

QLGA_HD i64 fx_join(Limb a) { return a.h * (i64(1) << 32) + a.l; }
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

// The potential's constants (those of PotConst, qlga_device.cuh) for the fixed-point form
struct FixPot {
    FxConst cphase, dz, dr, e0, R;
    float cphase_f, dz_f, dr_f, R_log;
    FixPot() = default;
    __host__ FixPot(double cphase_, double dz_, double dr_, double e0_, double R_)
        : cphase(cphase_), dz(dz_), dr(dr_), e0(e0_), R(R_), cphase_f(float(cphase_)), dz_f(float(dz_)), dr_f(float(dr_)),
          R_log(R_ == 0.0 ? -100000.f : float(std::log2(std::fabs(R_)))) {}
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
constexpr int kFxMinExp = 1022 - 930;
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

constexpr int kFxNone = -100000;  // the exponent of an empty level
constexpr int kFxFloor = -950;    // the smallest exponent of a level of a vector

// Bits of the larger of two integers' magnitudes (one's complement)
QLGA_HD int fx_bits_of(i64 a, i64 b) {
    const i64 m = (a ^ (a >> 63)) | (b ^ (b >> 63));
    return m ? 64 - fx_clz(m) : 0;
}
QLGA_HD int fx_max(int a, int b) { return a > b ? a : b; }
QLGA_HD int fx_clamp(int n, int lo, int hi) { return n < lo ? lo : (n > hi ? hi : n); }
QLGA_HD float fx_pow2f(int n) {  // 2^n, clamped to the normal range
    n = fx_clamp(n, -126, 127);
    union {
        unsigned u;
        float f;
    } p;
    p.u = unsigned(n + 127) << 23;
    return p.f;
}
// v 2^n for any n (the caller knows that it fits)
QLGA_HD i64 fx_scale_any(i64 v, int n) { return fx_scale(v, fx_max(n, -63)); }

// A field by levels: psi_m = (re, im) 2^(e - 58), the mantissas below 2^58 and the larger one in [2^57, 2^58)
struct FxLevels {
    FxVec p;
    int e[5];
};
QLGA_HD void fx_level(i64 re, i64 im, int unit, Limb& lr, Limb& li, int& e) {  // of (re, im) 2^unit, below 2^62
    const int b = fx_bits_of(re, im);
    lr = fx_split(fx_scale(re, 58 - b));
    li = fx_split(fx_scale(im, 58 - b));
    e = b ? unit + b : kFxNone;
}

// delta W of a site, between vectors whose level m is (re, im) 2^(T_m - 57): entry (m, j) times 2^(T_j - T_m), in
// 2^61 = 1.  The singlet term is conj(u_m) times the sum of v_j x_j (2^58 = 1).
struct FxW {
    Limb D[5];
    Limb upr[4], upi[4];  // row m + 1, from m: delta g1 c F_+
    Limb dnr[4], dni[4];  // row m, from m + 1: its conjugate
    FxVec u, v;
};

// t <- -i delta W t
QLGA_HD void fx_apply(const FxW& W, const FxVec& t, i64 ore[5], i64 oim[5]) {
    FxAcc tp = fx_zero<58>(), tn = {0, 0}, ti = fx_zero<58>();
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        fx_mac(tp, W.v.re[j], t.re[j]);
        fx_mac(tn, W.v.im[j], t.im[j]);
        fx_mac(ti, W.v.re[j], t.im[j]);
        fx_mac(ti, W.v.im[j], t.re[j]);
    }
    const Limb Gr = fx_split(fx_sum<58>(tp - tn)), Gi = fx_split(fx_sum<58>(ti));
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
        if (i > 0) {
            fx_mac(yr, W.upr[i - 1], t.re[i - 1]);
            fx_mac(nr, W.upi[i - 1], t.im[i - 1]);
            fx_mac(yi, W.upr[i - 1], t.im[i - 1]);
            fx_mac(yi, W.upi[i - 1], t.re[i - 1]);
        }
        if (i < 4) {  // the entry is the conjugate
            fx_mac(yr, W.dnr[i], t.re[i + 1]);
            fx_mac(yr, W.dni[i], t.im[i + 1]);
            fx_mac(yi, W.dnr[i], t.im[i + 1]);
            fx_mac(ni, W.dni[i], t.re[i + 1]);
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

constexpr float kFxNormMax = 1.f;  // of delta W between the scaled vectors
// Truncation of the Taylor sums, relative to the site: the same terms are missing from step to step, so
// the bound is a sixteenth of FP64's 2^-53 (a term of the FP32 part costs 2% of U).  Orders whose bound is
// above kFxTolF run in fixed point.
constexpr float kFxTol = 6.9388939e-18f;   // 2^-57
constexpr float kFxTolF = 4.6566129e-10f;  // 2^-31

// Smallest K with beta^(K+1)/(K+1)! <= tol (beta <= 1: at most 19 for 2^-57, 12 for 2^-31)
QLGA_HD int fx_degree(float beta, float tol) {
    int K = 0;
    float term = beta;
    while (term > tol && K < kFxDegree - 1) {
        ++K;
        term *= beta * fx_inv(K + 1);
    }
    return K;
}

// The same matrix in FP32
struct FxWF {
    float D[5];
    FxCpxF up[4], dn[4], u[5], v[5];
    QLGA_HD explicit FxWF(const FxW& W) {
        const float s58 = 3.4694470e-18f, s61 = 4.3368087e-19f;  // 2^-58, 2^-61
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            D[i] = fx_float(W.D[i], s61);
            u[i] = {fx_float(W.u.re[i], s61), fx_float(W.u.im[i], s61)};
            v[i] = {fx_float(W.v.re[i], s58), fx_float(W.v.im[i], s58)};
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            up[i] = {fx_float(W.upr[i], s61), fx_float(W.upi[i], s61)};
            dn[i] = {fx_float(W.dnr[i], s61), fx_float(W.dni[i], s61)};
        }
    }
};
QLGA_HD FxCpxF fx_dot_f(const FxWF& W, const FxCpxF t[5]) {
    FxCpxF a = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        a.re = fmaf(W.v[j].re, t[j].re, fmaf(-W.v[j].im, t[j].im, a.re));
        a.im = fmaf(W.v[j].re, t[j].im, fmaf(W.v[j].im, t[j].re, a.im));
    }
    return a;
}
// o <- (-i ik) delta W t, with the dot product of v and t
QLGA_HD void fx_apply_f(const FxWF& W, const FxCpxF t[5], FxCpxF g, FxCpxF o[5], float ik) {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        float yr = fmaf(W.D[i], t[i].re, fmaf(W.u[i].re, g.re, W.u[i].im * g.im));
        float yi = fmaf(W.D[i], t[i].im, fmaf(W.u[i].re, g.im, -W.u[i].im * g.re));
        if (i > 0) {
            const FxCpxF e = W.up[i - 1];
            yr = fmaf(e.re, t[i - 1].re, fmaf(-e.im, t[i - 1].im, yr));
            yi = fmaf(e.re, t[i - 1].im, fmaf(e.im, t[i - 1].re, yi));
        }
        if (i < 4) {
            const FxCpxF e = W.dn[i];
            yr = fmaf(e.re, t[i + 1].re, fmaf(e.im, t[i + 1].im, yr));
            yi = fmaf(e.re, t[i + 1].im, fmaf(-e.im, t[i + 1].re, yi));
        }
        o[i] = {ik * yi, -ik * yr};
    }
}

// The quadratic forms of psi: rho and F_z in units of 2^(en - 56), F_+ / 2 = (fr, fi) 2^(fe - 56) and
// delta g1 F_+ = (er, ei) 2^(ee - 60), the larger of the two in [2^59, 2^60) in magnitude.  Each is good to 2^-57 of the
// largest of its terms.
struct FxForms {
    i64 rho, Fz, fr, fi, er, ei;
    int en, fe, ee;
};
QLGA_HD void fx_coupled_spin(const FxConst& e0, FxForms& f) {  // (er, ei) from (fr, fi), below 2^60
    f.er = fx_mul_full<60>(e0.m, fx_split(f.fr));
    f.ei = fx_mul_full<60>(e0.m, fx_split(f.fi));
    const int b = fx_bits_of(f.er, f.ei);
    f.er = fx_scale(f.er, 60 - b);
    f.ei = fx_scale(f.ei, 60 - b);
    f.ee = b ? b + e0.ex + f.fe - 55 : kFxNone;
}

QLGA_HD void fx_forms(const FxLevels& psi, const FixPot& C, FxForms& f) {
    const Limb *re = psi.p.re, *im = psi.p.im;
    const int* e = psi.e;
    f.en = 2 * fx_max(fx_max(fx_max(e[0], e[1]), fx_max(e[2], e[3])), e[4]);
    i64 n[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {  // with l l': of a square it has no zero mean
        FxAcc s = fx_zero<60>();
        fx_mac(s, re[i], re[i]);
        fx_mac(s, im[i], im[i]);
        s.mid += (fx_mad(re[i].l, re[i].l, 0) >> 32) + (fx_mad(im[i].l, im[i].l, 0) >> 32);
        n[i] = fx_scale_any(fx_sum<60>(s), 2 * e[i] - f.en);
    }
    f.rho = (n[0] + n[1]) + (n[2] + n[3]) + n[4];
    f.Fz = 2 * (n[0] - n[4]) + (n[1] - n[3]);
    f.fe = fx_max(fx_max(e[0] + e[1], e[1] + e[2]), fx_max(e[2] + e[3], e[3] + e[4]));
    const Limb r = fx_split(kFxR32m1);
    f.fr = f.fi = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // c conj(psi_i) psi_{i+1}
        FxAcc a = fx_zero<60>(), b = fx_zero<60>(), c = {0, 0};
        fx_mac(a, re[i], re[i + 1]);
        fx_mac(a, im[i], im[i + 1]);
        fx_mac(b, re[i], im[i + 1]);
        fx_mac(c, im[i], re[i + 1]);
        const int sh = e[i] + e[i + 1] - f.fe;
        i64 x = fx_scale_any(fx_sum<60>(a), sh), y = fx_scale_any(fx_sum<60>(b - c), sh);
        if (i == 1 || i == 2) {
            x += fx_mul(r, fx_split(x));
            y += fx_mul(r, fx_split(y));
        }
        f.fr += x;
        f.fi += y;
    }
    fx_coupled_spin(C.e0, f);
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

// c q 2^unit in 2^61 = 1 (below 2^62 in the domain)
QLGA_HD i64 fx_coupled(const FxConst& c, i64 q, int unit) {
    return fx_scale(fx_mul_full<60>(c.m, fx_split(q)), fx_clamp(c.ex + unit + 61, -63, 30));
}

// Sizes as logarithms to base 2
constexpr float kFxLogNone = -100000.f;
QLGA_HD float fx_log2(float x) {
#ifdef __CUDA_ARCH__
    return __log2f(x);
#else
    return log2f(x);
#endif
}
QLGA_HD float fx_exp2(float x) {
#ifdef __CUDA_ARCH__
    return exp2f(x);
#else
    return ::exp2f(x);
#endif
}
QLGA_HD float fx_log_of(i64 re, i64 im, int e) {  // of |(re, im)| 2^e, 0: none (components below 2^62)
    const float a = 2.1684043e-19f * float(re), b = 2.1684043e-19f * float(im), q = fmaf(a, a, b * b);  // 2^-62
    return q > 0.f ? fmaf(0.5f, fx_log2(q), float(e + 62)) : kFxLogNone;
}

// What bounds the entries of delta W: log2 of |psi_m|, |delta g1 F_+| and |delta g2 / 5|
struct FxSizes {
    float p[5], e, R;
};
// log2 of the singlet term's row factor over |psi_{-m}|: |delta g2 / 5| sum_j |psi_{-j}| 2^L_j
QLGA_HD float fx_log_dot(const FxSizes& z, const float L[5]) {
    float g = z.p[4] + L[0];
#pragma unroll
    for (int j = 1; j < 5; ++j) g = fmaxf(g, z.p[4 - j] + L[j]);
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < 5; ++j) v += fx_exp2(z.p[4 - j] + L[j] - g);
    return z.R + g + fx_log2(v);
}
constexpr float kFxLogR32 = 0.29248125f;  // log2 sqrt(3/2)
QLGA_HD float fx_log_link(const FxSizes& z, int i) { return i == 0 || i == 3 ? z.e : z.e + kFxLogR32; }  // (i, i + 1)

// The exponents T of a vector's levels of sizes own (moduli below 2^T), raised until every entry of delta W off the
// diagonal times 2^(T_j - T_m) is below 2^-margin, or what the field itself allows: a weak level that a strong
// one drives takes a few times the size of what it receives in a step, which 2^-57 of still resolves
// better than FP64 does.  In most fields nothing changes.
QLGA_HD void fx_budget(const FxSizes& z, const float own[5], float margin, int T[5]) {
    float L[5], pm = z.p[0];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        L[m] = own[m];
        pm = fmaxf(pm, z.p[m]);
    }
    const float ke = fmaxf(0.f, fminf(margin, -kFxLogR32 - z.e)), ks = fmaxf(0.f, fminf(margin, -z.R - 2.f * pm));
#pragma unroll 1
    for (int it = 0; it < 8; ++it) {
        const float g = fx_log_dot(z, L) + ks;
        float N[5];
        bool raised = false;
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            N[m] = fmaxf(L[m], g + z.p[4 - m]);
            if (m < 4) N[m] = fmaxf(N[m], fx_log_link(z, m) + ke + L[m + 1]);
            if (m > 0) N[m] = fmaxf(N[m], fx_log_link(z, m - 1) + ke + L[m - 1]);
            raised = raised || N[m] > L[m] + 0.01f;
        }
        if (!raised) break;
#pragma unroll
        for (int m = 0; m < 5; ++m) L[m] = N[m];
    }
#pragma unroll
    for (int m = 0; m < 5; ++m) T[m] = int(ceilf(L[m] + 0.001f));
}
// The exponent of the dot product of v and a vector
QLGA_HD int fx_dot_exp(const int P[5], const int T[5]) {
    return fx_max(fx_max(fx_max(P[4] + T[0], P[0] + T[4]), fx_max(P[3] + T[1], P[1] + T[3])), P[2] + T[2]);
}

// A bound of the scaled matrix: the largest row sum of the moduli, which bounds every Taylor term of a vector with
// moduli of at most one.  Not finite, or large, where the entries would not fit their integers.
QLGA_HD float fx_norm(const FxSizes& z, const FxForms& f, const FixPot& C, const int T[5]) {
    const float un = fx_pow2f(f.en - 56);
    const float gz = C.dz_f * un * float(f.Fz), g2r = C.dr_f * un * float(f.rho);
    float L[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) L[m] = float(T[m]);
    const float g = fx_log_dot(z, L);
    float w = 0.f;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        float row = fabsf(fmaf(float(2 - m), gz, -g2r)) + fx_exp2(g + z.p[4 - m] - L[m]);
        if (m < 4) row += fx_exp2(fx_log_link(z, m) + L[m + 1] - L[m]);
        if (m > 0) row += fx_exp2(fx_log_link(z, m - 1) + L[m - 1] - L[m]);
        w = row > w || !(row == row) ? row : w;
    }
    return 1.0001f * w;
}

// The exponents and the norm: a margin of 1 bit, up to 2 for a field too dense for it (a bit of the margin costs a
// driven level one)
constexpr int kFxMargins = 3;
QLGA_HD float fx_margin(int k) { return 1.f + 0.5f * float(k); }
QLGA_HD float fx_exponents(const FxSizes& z, const FxForms& f, const FixPot& C, const float own[5], int T[5]) {
    float w = 0.f;
#pragma unroll 1
    for (int k = 0; k < kFxMargins; ++k) {
        fx_budget(z, own, fx_margin(k), T);
        w = fx_norm(z, f, C, T);
        if (w <= kFxNormMax) break;
    }
    return w;
}

QLGA_HD void fx_build_w(const FxLevels& psi, const FxForms& f, const FixPot& C, const int T[5], FxW& W) {
    const i64 gz = fx_coupled(C.dz, f.Fz, f.en - 56), g2r = fx_coupled(C.dr, f.rho, f.en - 56);
#pragma unroll
    for (int i = 0; i < 5; ++i) W.D[i] = fx_split((2 - i) * gz - g2r);
    const Limb r = fx_split(kFxR32m1);
    const i64 er1 = f.er + fx_mul(r, fx_split(f.er)), ei1 = f.ei + fx_mul(r, fx_split(f.ei));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const i64 er = i == 0 || i == 3 ? f.er : er1, ei = i == 0 || i == 3 ? f.ei : ei1;
        const int up = fx_clamp(f.ee + T[i] - T[i + 1] + 1, -63, 2), dn = fx_clamp(f.ee + T[i + 1] - T[i] + 1, -63, 2);
        W.upr[i] = fx_split(fx_scale(er, up));
        W.upi[i] = fx_split(fx_scale(ei, up));
        W.dnr[i] = fx_split(fx_scale(er, dn));
        W.dni[i] = fx_split(fx_scale(ei, dn));
    }
    const int g = fx_dot_exp(psi.e, T);
#pragma unroll
    for (int j = 0; j < 5; ++j) {  // u_j = (-1)^j psi_{4-j}
        const Limb pr = psi.p.re[4 - j], pi = psi.p.im[4 - j];
        const int sv = fx_clamp(psi.e[4 - j] + T[j] - g, -63, 0), su = fx_clamp(C.R.ex + psi.e[4 - j] + g - T[j] + 3, -63, 5);
        i64 vr = fx_scale(fx_join(pr), sv), vi = fx_scale(fx_join(pi), sv);
        i64 ur = fx_scale(fx_mul_full<60>(C.R.m, pr), su), ui = fx_scale(fx_mul_full<60>(C.R.m, pi), su);
        if (j & 1) {
            vr = -vr;
            vi = -vi;
            ur = -ur;
            ui = -ui;
        }
        W.v.re[j] = fx_split(vr);
        W.v.im[j] = fx_split(vi);
        W.u.re[j] = fx_split(ur);
        W.u.im[j] = fx_split(ui);
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
QLGA_HD int fx_warp_max(int v) {
#ifdef __CUDA_ARCH__
    return __reduce_max_sync(0xffffffffu, v);
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

// A bound of a modulus from the largest high limb of its components, which are in 2^57 = 1
QLGA_HD float fx_size(int h) { return 4.2146848e-8f * float(h + 1); }  // sqrt(2) 2^-25
QLGA_HD int fx_abs_limb(Limb a) { return a.h < 0 ? -a.h : a.h; }
QLGA_HD float fx_size(const FxVec& t) {
    int h = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) h = fx_max(h, fx_max(fx_abs_limb(t.re[i]), fx_abs_limb(t.im[i])));
    return fx_size(h);
}

// x <- exp(-i delta W) x for one vector, w >= the warp's norm of W: the terms T_k / k! in fixed point until the next one
// is below 2^-31, then in FP32 until it is below 2^-57.  A term is bounded by w times the one before it; the sizes of the
// terms themselves decide, since a scaled norm is two to five times what they shrink by (bounds of w^k / k! alone
// took one more order in fixed point, a fifth of U).
QLGA_HD void fx_taylor(const FxW& W, i64 re[5], i64 im[5], float w) {
    FxVec t;
    i64 tr[5], ti[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        t.re[i] = fx_split(re[i]);
        t.im[i] = fx_split(im[i]);
    }
    float q = fx_warp_max(fx_size(t));  // of T_k / k!
    int k = 0;
    float fact = 6.9388939e-18f;  // 2^-57 / k!
#pragma unroll 1
    while (w * q * fx_inv(k + 1) > kFxTolF && k < kFxTerms) {
        ++k;
        fact *= fx_inv(k);
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
        q = 1.4411519e17f * fact * fx_warp_max(fx_size(t));  // 2^57
    }
    q *= w * fx_inv(k + 1);
    if (q > kFxTol) {
        FxCpxF tf[5], sf[5], of[5];
        const FxWF Wf(W);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            tf[i] = {fx_float(t.re[i], fact), fx_float(t.im[i], fact)};
            sf[i] = {0.f, 0.f};
        }
#pragma unroll 1
        while (q > kFxTol && k < kFxDegree - 1) {
            ++k;
            fx_apply_f(Wf, tf, fx_dot_f(Wf, tf), of, fx_inv(k));
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                tf[i] = of[i];
                sf[i] = {sf[i].re + of[i].re, sf[i].im + of[i].im};
            }
            q *= w * fx_inv(k + 1);
        }
        const float one = 144115188075855872.f;  // 2^57
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

// e^{-i theta} - 1 = (-c, -s) for a theta of any size (fields denser than |theta| = 1/4 are rare)
static __host__ __device__ __noinline__ void fx_phase_large(double theta, i64* c, i64* s) {
    double sn, cs;
    sincos(theta, &sn, &cs);
    *c = i64(rint((1.0 - cs) * 2305843009213693952.0));
    *s = i64(rint(sn * 2305843009213693952.0));
}

// e^{-i theta} - 1 = (-c, -s) of a site from its density rho 2^unit, for a warp with a lane beyond |theta| = 1/4 in FP64
QLGA_HD void fx_site_phase(i64 rho, int unit, const FixPot& C, i64& c, i64& s) {
    const float theta = fabsf(C.cphase_f) * fx_pow2f(unit) * float(rho);
    if (!fx_warp_all(theta <= 0.25f)) {
        const double th = ldexp(double(C.cphase.m.h) * 4294967296.0 + double(C.cphase.m.l), C.cphase.ex - 60 + fx_max(unit, -960)) * double(rho);
        fx_phase_large(th, &c, &s);
    } else {
        fx_phase(fx_coupled(C.cphase, rho, unit), c, s);
    }
}

// U on one site of a warp.  In: level m of psi and d as integers below 2^62 of unit 2^e[m], `true` amplitudes
// 2^in_log2 times that; ok = false: a lane whose input has no such form.  Out: (psi', d') =
// (U psi, U d) as integers of the units 2^e[m], below 2^60.  Returns false, with
// nothing changed, if a lane of the warp lies outside the domain.  All 32 lanes take part: the
// orders of the Taylor sums are those of the warp's largest norm.
QLGA_HD bool fx_unitary(i64 pr[5], i64 pi[5], i64 dr[5], i64 di[5], int e[5], int in_log2, bool ok, const FixPot& C) {
    FxLevels psi;
    FxSizes z;
    float L[5];  // sizes of the levels of both vectors
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        fx_level(pr[i], pi[i], e[i] + in_log2, psi.p.re[i], psi.p.im[i], psi.e[i]);
        z.p[i] = fx_log_of(pr[i], pi[i], e[i] + in_log2);
        L[i] = fmaxf(fmaxf(z.p[i], fx_log_of(dr[i], di[i], e[i] + in_log2)), float(kFxFloor));
    }
    FxForms f;
    fx_forms(psi, C, f);
    z.e = fx_log_of(f.er, f.ei, f.ee - 60);
    z.R = C.R_log;
    int T[5];
    const float w = fx_exponents(z, f, C, L, T);
    ok = ok && w <= kFxNormMax;
    if (!fx_warp_all(ok)) return false;
    const float wmax = fx_warp_max(w);
    FxW W;
    fx_build_w(psi, f, C, T, W);
    i64 pc, ps;
    fx_site_phase(f.rho, f.en - 56, C, pc, ps);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int n = fx_clamp(e[i] + in_log2 + 57 - T[i], -63, 57);
        pr[i] = fx_scale(pr[i], n);
        pi[i] = fx_scale(pi[i], n);
        dr[i] = fx_scale(dr[i], n);
        di[i] = fx_scale(di[i], n);
        e[i] = T[i] - in_log2 - 57;
    }
#pragma unroll 1
    for (int v = 0; v < 2; ++v) {  // one copy of the code for both vectors
        fx_taylor(W, pr, pi, wmax);
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
    return true;
}

// The biased exponent of a level whose largest high word is m, and whether integers can hold it: finite, below
// 2^60, and not between nothing and 2^-930
QLGA_HD int fx_level_exponent(unsigned m, bool& ok) {
    ok = ok && m < (unsigned(1023 + 60) << 20) && (m == 0 || m >= (unsigned(kFxMinExp + 1) << 20));
    return fx_exponent(m);
}

// U on the pair (a, b) of one site of a warp in FP64, by fx_unitary; the arguments are those of
// potential_site, with in_log2 = -log2 sigma and out_log2 = log2 out_scale.  PQ: (a, b) become
// (P, Q) = (a + i b, a - i b) of the result, summed before the conversion.  Returns false, with nothing changed, outside the domain.
template <bool PQ>
QLGA_HD bool fx_potential(double ar[5], double ai[5], double br[5], double bi[5], int in_log2,
                                             int out_log2, const FixPot& C) {
    bool ok = true;
    int e[5];
    i64 pr[5], pi[5], dr[5], di[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int E = fx_level_exponent(fx_top(fx_top(fx_top(fx_top(0, ar[i]), ai[i]), br[i]), bi[i]), ok);
        e[i] = E - 1022 - 60;
        const i64 a0 = fx_from_double<60>(ar[i], E), a1 = fx_from_double<60>(ai[i], E);
        const i64 b0 = fx_from_double<60>(br[i], E), b1 = fx_from_double<60>(bi[i], E);
        pr[i] = a0 + b0;
        pi[i] = a1 + b1;
        dr[i] = a0 - b0;
        di[i] = a1 - b1;
    }
    if (!fx_unitary(pr, pi, dr, di, e, in_log2, ok, C)) return false;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const FxToDouble to(e[i] + out_log2);
        const i64 a0 = pr[i] + dr[i], a1 = pi[i] + di[i], b0 = pr[i] - dr[i], b1 = pi[i] - di[i];
        ar[i] = to(PQ ? a0 - b1 : a0);
        ai[i] = to(PQ ? a1 + b0 : a1);
        br[i] = to(PQ ? a0 + b1 : b0);
        bi[i] = to(PQ ? a1 - b0 : b1);
    }
    return true;
}

}  // namespace qlga
