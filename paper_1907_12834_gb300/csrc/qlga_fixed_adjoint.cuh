// qlga_fixed_adjoint.cuh -- the pull-back through U at a site in integer fixed point.
//
// The FP64 pull-back (qlga_adjoint.cuh) is 2250 FP64 instructions a site in its sweeps alone, one every 66 cycles
// (qlga_fixed.cuh).  Here both sweeps run on the numbers of fx_unitary: W, the phase and the vectors psi = a + b, d = a - b
// with one exponent; the cotangents ga + gb and ga - gb with another.
// Orders whose bound is below 2^-31 run in FP32, as
// there.  256^2 (g = (1, 0.1, 1)): 0.186 ms for the x axis of K^dagger and the pull-back, 0.053 of them the FP64 stencil,
// against 0.464 with FP64 sweeps; a gradient of 12 steps 5.2 ms against 8.5, its error against 64 bits 3.5e-15 against 3.3e-15
// (4.0e-15 with the Frechet recursions before).
//
// Magnitudes.  Vectors and cotangents are below 2^57 in each component (vectors 2^56, so that every v_k is), and W's sums fit
// as for d in fx_unitary.
#pragma once

#include "qlga_adjoint.cuh"
#include "qlga_fixed.cuh"

namespace qlga {

constexpr int kFxAdjSlots = 8;  // beta <= 1/4: at most 8 orders in fixed point

struct FxAdjSlot {
    i64 re[5], im[5];
};

// 1/k in 2^61 = 1
struct FxInvInt {
    int h[kFxAdjSlots + 1], l[kFxAdjSlots + 1];
};
constexpr FxInvInt make_fx_inv_int() {
    FxInvInt t{};
    for (int k = 1; k <= kFxAdjSlots; ++k) {
        const i64 v = fx_ratio(1, k), h = (v + (i64(1) << 31)) >> 32;
        t.h[k] = int(h);
        t.l[k] = int(v - h * (i64(1) << 32));
    }
    return t;
}
__constant__ FxInvInt c_fx_inv_int = make_fx_inv_int();

// out <- -i delta W t
__device__ __forceinline__ void fx_apply_ints(const FxW& W, const i64 re[5], const i64 im[5], i64 ore[5], i64 oim[5]) {
    FxVec t;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        t.re[i] = fx_split(re[i]);
        t.im[i] = fx_split(im[i]);
    }
    fx_apply(W, t, ore, oim);
}

// 2^e, 0 below the normal range (a site or a cotangent of nothing)
__device__ __forceinline__ double fx_pow2_or_0(int e) { return e < -1022 ? 0.0 : fx_pow2(min(e, 1023)); }

// Sums of the reverse sweep, as AdjSweep: products of a cotangent and a vector over 2^60 (s: of u . mu and u . v)
struct FxAdjSums {
    i64 upr[2], upi[2], dnr[2], dni[2], z1, z2, qr[5], qi[5], s, tau;
};

struct LimbC {
    Limb re, im;
};
QLGA_HD LimbC fx_limbs(i64 re, i64 im) { return {fx_split(re), fx_split(im)}; }
// a limb of -2^31 has no negative: one unit off
QLGA_HD Limb fx_neg(Limb a) { return {-a.h, -(a.l > -0x7fffffff ? a.l : -0x7fffffff)}; }
// s += Re / Im of conj(a) b
QLGA_HD void fx_conj_mac(FxAcc& re, FxAcc& im, LimbC a, LimbC b) {
    fx_mac(re, a.re, b.re);
    fx_mac(re, a.im, b.im);
    fx_mac(im, a.re, b.im);
    fx_mac(im, fx_neg(a.im), b.re);
}

// The contractions of mu with v; (ur, ui) = u
__device__ __forceinline__ void fx_contract(FxAdjSums& S, const i64 ur_[5], const i64 ui_[5], const i64 mr[5],
                                            const i64 mi[5], const FxAdjSlot& h) {
    auto dot = [&](const i64 re[5], const i64 im[5]) {  // u . vector / 2^60
        FxAcc a = fx_zero<60>(), b = fx_zero<60>();
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const LimbC u = fx_limbs(ur_[i], ui_[i]), x = fx_limbs(re[i], im[i]);
            fx_mac(a, u.re, x.re);
            fx_mac(a, fx_neg(u.im), x.im);
            fx_mac(b, u.re, x.im);
            fx_mac(b, u.im, x.re);
        }
        return fx_limbs(fx_sum<60>(a), fx_sum<60>(b));
    };
    const LimbC p = dot(mr, mi), t = dot(h.re, h.im);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const LimbC m = fx_limbs(mr[i], mi[i]), v = fx_limbs(h.re[i], h.im[i]);
        if (i < 4) {
            const LimbC m1 = fx_limbs(mr[i + 1], mi[i + 1]), v1 = fx_limbs(h.re[i + 1], h.im[i + 1]);
            const int c = i == 0 || i == 3 ? 0 : 1;
            FxAcc ur = fx_zero<60>(), ui = fx_zero<60>(), wr = fx_zero<60>(), wi = fx_zero<60>();
            fx_conj_mac(ur, ui, m, v1);
            fx_conj_mac(wr, wi, m1, v);
            S.upr[c] += fx_sum<60>(ur);
            S.upi[c] += fx_sum<60>(ui);
            S.dnr[c] += fx_sum<60>(wr);
            S.dni[c] += fx_sum<60>(wi);
        }
        if (i != 2) {
            FxAcc z = fx_zero<60>();  // Im conj(mu_i) v_i
            fx_mac(z, m.re, v.im);
            fx_mac(z, fx_neg(m.im), v.re);
            const i64 w = fx_sum<60>(z);
            if (i == 0) S.z2 += w;
            else if (i == 1) S.z1 += w;
            else if (i == 3) S.z1 -= w;
            else S.z2 -= w;
        }
        // conj(p) v - conj(t) mu
        FxAcc qr = fx_zero<60>(), qi = fx_zero<60>();
        fx_conj_mac(qr, qi, p, v);
        const LimbC nm = {fx_neg(m.re), fx_neg(m.im)};
        fx_conj_mac(qr, qi, t, nm);
        S.qr[i] += fx_sum<60>(qr);
        S.qi[i] += fx_sum<60>(qi);
    }
    FxAcc sr = fx_zero<60>(), si = fx_zero<60>();
    fx_conj_mac(sr, si, p, t);
    S.s += fx_sum<60>(si);
}

// v / k
QLGA_HD i64 fx_div(i64 v, Limb ik) { return fx_mul(ik, fx_split(v)); }

// The pull-back at a site of a warp; the arguments are those of potential_vjp_site.  Returns false, with nothing
// changed, outside the domain (that of fx_unitary, and cotangents below 2^400).  All 32 lanes take part.
__device__ __forceinline__ bool fx_vjp_site(const cpx<double> a[5], const cpx<double> b[5], cpx<double> ga[5],
                                            cpx<double> gb[5], const AdjConst<double>& A, double dc[3]) {
    const FixPot& C = A.pc.fx;
    unsigned mx = 0, mg = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        auto hi = [](double x) { return fx_hi(x) & 0x7fffffffu; };
        mx = max(mx, max(max(hi(a[i].re), hi(a[i].im)), max(hi(b[i].re), hi(b[i].im))));
        mg = max(mg, max(max(hi(ga[i].re), hi(ga[i].im)), max(hi(gb[i].re), hi(gb[i].im))));
    }
    bool ok = mx < (unsigned(1023 + 60) << 20) && mg < (unsigned(1023 + 400) << 20);
    const int Ex = fx_exponent(mx), Eg = fx_exponent(mg);
    i64 xr[5], xi[5], yr[5], yi[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const i64 a0 = fx_from_double<60>(a[i].re, Ex), a1 = fx_from_double<60>(a[i].im, Ex);
        const i64 b0 = fx_from_double<60>(b[i].re, Ex), b1 = fx_from_double<60>(b[i].im, Ex);
        xr[i] = a0 + b0;
        xi[i] = a1 + b1;
        yr[i] = a0 - b0;
        yi[i] = a1 - b1;
    }
    int ex = Ex - 1022 - 60, eg = Eg - 1022 - 60;
    const int np = fx_headroom(xr, xi);
    FxVec p;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        p.re[i] = fx_split(fx_shift(xr[i], np));
        p.im[i] = fx_split(fx_shift(xi[i], np));
    }
    FxForms f;
    fx_forms(p, f);
    const int et = ex + np;
    const FxBounds bd = fx_bounds(f, et, C);
    ok = ok && bd.beta <= kFxBetaMax;
    if (!__all_sync(0xffffffffu, ok)) return false;
    const float beta = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(bd.beta)));
    const int K = fx_degree(beta, kFxTol);
    const int kA = max(1, min(K, fx_degree(beta, kFxTolF) + 1));  // beta^kA / kA! <= 2^-31
    FxW W;
    fx_build_w(p, f, et, C, W);
    i64 pc, ps;
    fx_site_phase(f.rho, et, bd.theta, C, pc, ps);

    i64 gr[5], gi[5], hr[5], hi[5];  // ga + gb, then ga - gb
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const i64 a0 = fx_from_double<60>(ga[i].re, Eg), a1 = fx_from_double<60>(ga[i].im, Eg);
        const i64 b0 = fx_from_double<60>(gb[i].re, Eg), b1 = fx_from_double<60>(gb[i].im, Eg);
        gr[i] = a0 + b0;
        gi[i] = a1 + b1;
        hr[i] = a0 - b0;
        hi[i] = a1 - b1;
    }
    i64 ur[5], ui[5];  // u_j = (-1)^j psi_{4-j}
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const i64 re = fx_shift(xr[4 - j], np), im = fx_shift(xi[4 - j], np);
        ur[j] = (j & 1) ? -re : re;
        ui[j] = (j & 1) ? -im : im;
    }
    const int nx = max(np, fx_headroom(yr, yi)) + 2, ng = max(fx_headroom(gr, gi), fx_headroom(hr, hi)) + 1;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        xr[i] = fx_shift(xr[i], nx);
        xi[i] = fx_shift(xi[i], nx);
        yr[i] = fx_shift(yr[i], nx);
        yi[i] = fx_shift(yi[i], nx);
        gr[i] = fx_shift(gr[i], ng);
        gi[i] = fx_shift(gi[i], ng);
        hr[i] = fx_shift(hr[i], ng);
        hi[i] = fx_shift(hi[i], ng);
    }
    ex += nx;
    eg += ng;

    FxAdjSums S;
#pragma unroll
    for (int i = 0; i < 2; ++i) S.upr[i] = S.upi[i] = S.dnr[i] = S.dni[i] = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) S.qr[i] = S.qi[i] = 0;
    S.z1 = S.z2 = S.s = S.tau = 0;
    AdjSweep<float> F;  // the FP32 steps' share, vectors and cotangents in 2^57 = 1
    F.clear();
    const float s58 = 3.4694470e-18f, s57 = 6.9388939e-18f, s61 = 4.3368087e-19f;  // 2^-58, 2^-57, 2^-61
    WOp<float> Wf;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        Wf.D[i] = fx_float(W.D[i], s61);
        Wf.u[i] = {fx_float(W.u.re[i], s58), fx_float(W.u.im[i], s58)};
    }
    Wf.ep[0] = Wf.ep[3] = {fx_float(W.e0r, s61), fx_float(W.e0i, s61)};
    Wf.ep[1] = Wf.ep[2] = {fx_float(W.e1r, s61), fx_float(W.e1i, s61)};
    Wf.R = W.Rf;
    auto op_f = [&](i64 v) { return fx_float(fx_split(v), s57); };
    FxAdjSlot kept[kFxAdjSlots];
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {  // one copy of the code for both vectors
        fx_rotate(pc, -ps, gr, gi);  // lambda_0 = e^{i theta} g
        // forward sweep
        i64 vr[5], vi[5];
        cpx<float> xf[5], vf[5];
        HornerSlot<float> keptf[kAdjSlotsF];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            vr[i] = xr[i];
            vi[i] = xi[i];
        }
        if (K > kA) {  // warp-uniform
#pragma unroll
            for (int i = 0; i < 5; ++i) vf[i] = xf[i] = {op_f(xr[i]), op_f(xi[i])};
#pragma unroll 1
            for (int k = K;; --k) {
                HornerSlot<float> h;
#pragma unroll
                for (int i = 0; i < 5; ++i) h.v[i] = vf[i];
                h.dot = singlet_dot(Wf, vf);
                if (k - kA <= kAdjSlotsF) keptf[k - kA - 1] = h;
                cpx<float> w[5];
                apply_dotted(Wf, vf, h.dot, w);
                const float ik = fx_inv(k);
                if (k == kA + 1) {
                    const float one = 144115188075855872.f * ik;  // 2^57 / k
                    auto whole = [](float x) {  // |x| < 2^57
                        const int top = fx_rint(x * 1.4901161e-8f);  // 2^-26
                        return (i64(top) << 26) + fx_rint(fmaf(float(top), -67108864.f, x));
                    };
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        vr[i] += whole(w[i].im * one);
                        vi[i] -= whole(w[i].re * one);
                    }
                    break;
                }
                horner_down(xf, w, vf, ik);
            }
        }
#pragma unroll 1
        for (int k = kA; k >= 1; --k) {
            FxAdjSlot& h = kept[k - 1];
            i64 wr[5], wi[5];
            fx_apply_ints(W, vr, vi, wr, wi);
            const Limb ik = {c_fx_inv_int.h[k], c_fx_inv_int.l[k]};
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                h.re[i] = vr[i];
                h.im[i] = vi[i];
                vr[i] = xr[i] + fx_div(wr[i], ik);
                vi[i] = xi[i] + fx_div(wi[i], ik);
            }
        }
        {  // tau += Im lambda_0^dagger v_0
            FxAcc t = fx_zero<60>();
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                fx_mac(t, fx_split(gr[i]), fx_split(vi[i]));
                fx_mac(t, fx_neg(fx_split(gi[i])), fx_split(vr[i]));
            }
            S.tau += fx_sum<60>(t);
        }
        // reverse sweep; (gr, gi) becomes the sum of the lambda_k
        i64 lr[5], li[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            lr[i] = gr[i];
            li[i] = gi[i];
        }
#pragma unroll 1
        for (int k = 1; k <= kA; ++k) {
            const Limb ik = {c_fx_inv_int.h[k], c_fx_inv_int.l[k]};
            i64 wr[5], wi[5];
            if (k > 1) {
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    lr[i] = fx_div(lr[i], ik);
                    li[i] = fx_div(li[i], ik);
                }
            }
            fx_apply_ints(W, lr, li, wr, wi);
            fx_contract(S, ur, ui, lr, li, kept[k - 1]);
#pragma unroll
            for (int i = 0; i < 5; ++i) {  // lambda_k = i W mu = -(-i W mu)
                lr[i] = -wr[i];
                li[i] = -wi[i];
                gr[i] += lr[i];
                gi[i] += li[i];
            }
        }
        if (K > kA) {
            cpx<float> lf[5], sf[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                lf[i] = {op_f(lr[i]), op_f(li[i])};
                sf[i] = {0.f, 0.f};
            }
#pragma unroll 1
            for (int k = kA + 1; k <= K; ++k) {
                HornerSlot<float> h;
                if (k - kA <= kAdjSlotsF) {
                    h = keptf[k - kA - 1];
                } else {
                    WOp<float> Wc = Wf;
                    cpx<float> xc[5];
                    HornerSlot<float> hc;
                    for (int i = 0; i < 5; ++i) xc[i] = xf[i];
                    horner_again<float>(&Wc, xc, K, k, &hc);
                    h = hc;
                }
                reverse_step(Wf, lf, h, fx_inv(k), F);
#pragma unroll
                for (int i = 0; i < 5; ++i) sf[i] = sf[i] + lf[i];
            }
            const float one = 144115188075855872.f;  // 2^57; the sum is below 2^-31
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                gr[i] += fx_rint(sf[i].re * one);
                gi[i] += fx_rint(sf[i].im * one);
            }
        }
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            xr[i] = yr[i];
            xi[i] = yi[i];
            const i64 tr = gr[i], ti = gi[i];
            gr[i] = hr[i];
            gi[i] = hi[i];
            hr[i] = tr;
            hi[i] = ti;
        }
    }
    // The sums are of psi with ga + gb and of d with ga - gb: twice those of a with ga and b with gb.  q has one factor
    // u and s two, in units of 2^(ex0 + np) where ex0 is psi's.
    const int ep = ex + eg + 60 - 1;  // unit of a product
    const double up = fx_pow2_or_0(ep), uf = up * 18014398509481984.0;  // FP32 part: 2^114 / 2^60 = 2^54 units
    auto join = [&](i64 v, float w) { return fma(double(w), uf, double(v) * up); };
    const double r32 = 1.2247448713915890491;
    const double upr = fma(r32, join(S.upr[1], F.up[1].re), join(S.upr[0], F.up[0].re));
    const double upi = fma(r32, join(S.upi[1], F.up[1].im), join(S.upi[0], F.up[0].im));
    const double dnr = fma(r32, join(S.dnr[1], F.dn[1].re), join(S.dnr[0], F.dn[0].re));
    const double dni = fma(r32, join(S.dni[1], F.dn[1].im), join(S.dni[0], F.dn[0].im));
    const double phx = upi + dni, phy = dnr - upr;
    const double phz = fma(2.0, join(S.z2, F.z2), join(S.z1, F.z1));
    const double tau = double(S.tau) * up;
    // q: p and t carry u / 2^60 (u in units of 2^et), FP32: u in 2^58 = 1
    const double uq = fx_pow2_or_0(et + 60) * up, ufq = uf * fx_pow2_or_0(et + 58);
    // s: a product over 2^60 of two u . vector / 2^60; FP32: (2^58 u)^2 2^114
    const double us = fx_pow2_or_0(2 * et + 120) * up, ufs = fx_pow2_or_0(2 * et + 116) * uf;
    cpx<double> psi[5], h[5];
    const double t0 = 2.0 * A.dg0 * tau, t1 = 2.0 * A.dg1;
    const cpx<double> lower = {t1 * phx, t1 * phy};
#pragma unroll
    for (int i = 0; i < 5; ++i) psi[i] = a[i] + b[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const double sg = (i & 1) ? -A.dg2_5 : A.dg2_5;
        const double qr = fma(double(F.q[4 - i].re), ufq, double(S.qr[4 - i]) * uq);
        const double qi = fma(double(F.q[4 - i].im), ufq, double(S.qi[4 - i]) * uq);
        h[i] = fma(double(2 - i), t1 * phz, t0) * psi[i];
        h[i] = {fma(sg, qi, h[i].re), fma(sg, qr, h[i].im)};  // i conj(q)
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const cpx<double> l = spin_c<double>(i) * lower;
        h[i] = cfmac(l, psi[i + 1], h[i]);
        h[i + 1] = cfma(l, psi[i], h[i + 1]);
    }
    const double uu = fx_pow2_or_0(2 * et + 60), rho = double(f.rho) * uu, Fz = double(f.Fz) * uu;
    const double Fpr = 2.0 * double(f.Fpr) * uu, Fpi = 2.0 * double(f.Fpi) * uu;
    dc[0] = A.delta * rho * tau;
    dc[1] = A.delta * (Fpr * phx + Fpi * phy + Fz * phz);
    dc[2] = A.delta * fma(double(F.s), ufs, double(S.s) * us) / 5.0;
    // U^dagger of the cotangents: half the sum and the difference
    const FxToDouble to(eg - 1);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        ga[i] = {to(gr[i] + hr[i]) + h[i].re, to(gi[i] + hi[i]) + h[i].im};
        gb[i] = {to(gr[i] - hr[i]) + h[i].re, to(gi[i] - hi[i]) + h[i].im};
    }
    return true;
}

}  // namespace qlga
