// qlga_fixed_adjoint.cuh -- the pull-back through U at a site in integer fixed point.
//
// The FP64 pull-back (qlga_adjoint.cuh) is 2250 FP64 instructions a site in its sweeps alone, one every 66 cycles
// (qlga_fixed.cuh).  Here both sweeps run on the numbers of fx_unitary: the vectors psi = a + b and d = a - b with an
// exponent T to a level, the cotangents ga + gb and ga - gb with their own, G, and delta W once between vectors
// of either scale.  Orders whose bound is below 2^-31 run in FP32, as there.  A gradient of 12 steps of 256^2 7.5 ms (8.3 with FP64
// sweeps), its error against 64 bits 2.7e-15 (3.3e-15).
//
// Magnitudes.  Vectors have moduli below 2^56 and cotangents below 2^57 of their levels' units, and grow by less
// than e along the sweeps.  Every sum of products carries the exponent of its largest term.
#pragma once

#include "qlga_adjoint.cuh"
#include "qlga_fixed.cuh"

namespace qlga {

constexpr int kFxAdjSlots = 13;  // norms up to 1: at most 13 orders in fixed point

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

// The exponents of the sums of the reverse sweep: a product of level i of a cotangent and j of a vector has G_i + T_j
struct FxAdjExp {
    int T[5], G[5], dT, dG;  // of the levels; of the dot products of v with a vector and a cotangent
    int xy, z, tau, q[5];
    __device__ __forceinline__ void sums() {
        xy = max(G[0] + T[1], G[1] + T[0]);
        tau = G[0] + T[0];
#pragma unroll
        for (int i = 1; i < 5; ++i) {
            if (i < 4) xy = max(xy, max(G[i] + T[i + 1], G[i + 1] + T[i]));
            tau = max(tau, G[i] + T[i]);
        }
        z = max(max(G[0] + T[0], G[1] + T[1]), max(G[3] + T[3], G[4] + T[4]));
#pragma unroll
        for (int i = 0; i < 5; ++i) q[i] = max(dG + T[i], dT + G[i]);
    }
};

// Sums of the reverse sweep, as AdjSweep: products over 2^60, in units of 2^(exponent - 53).  c_i is in up and dn, m in z.
struct FxAdjSums {
    i64 upr, upi, dnr, dni, z, qr[5], qi[5], s, tau;
};

struct LimbC {
    Limb re, im;
};
QLGA_HD LimbC fx_limbs(i64 re, i64 im) { return {fx_split(re), fx_split(im)}; }
// conj(a) b / 2^60
QLGA_HD void fx_conj_mul(LimbC a, LimbC b, i64& re, i64& im) {
    FxAcc r = fx_zero<60>(), i = fx_zero<60>(), n = {0, 0};
    fx_mac(r, a.re, b.re);
    fx_mac(r, a.im, b.im);
    fx_mac(i, a.re, b.im);
    fx_mac(n, a.im, b.re);
    re = fx_sum<60>(r);
    im = fx_sum<60>(i - n);
}
QLGA_HD i64 fx_conj_mul_im(LimbC a, LimbC b) {
    i64 re, im;
    fx_conj_mul(a, b, re, im);
    return im;
}
// The dot product of v and a vector
__device__ __forceinline__ LimbC fx_dot(const FxW& W, const i64 re[5], const i64 im[5]) {
    FxAcc a = fx_zero<58>(), n = {0, 0}, b = fx_zero<58>();
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const LimbC x = fx_limbs(re[i], im[i]);
        fx_mac(a, W.v.re[i], x.re);
        fx_mac(n, W.v.im[i], x.im);
        fx_mac(b, W.v.re[i], x.im);
        fx_mac(b, W.v.im[i], x.re);
    }
    return fx_limbs(fx_sum<58>(a - n), fx_sum<58>(b));
}

// The contractions of the cotangent mu with the vector v
__device__ __forceinline__ void fx_contract(FxAdjSums& S, const FxAdjExp& E, const FxW& WT, const FxW& WG, const i64 mr[5],
                                            const i64 mi[5], const FxAdjSlot& h) {
    const LimbC p = fx_dot(WG, mr, mi), t = fx_dot(WT, h.re, h.im);
    const Limb r32m1 = fx_split(kFxR32m1);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const LimbC m = fx_limbs(mr[i], mi[i]), v = fx_limbs(h.re[i], h.im[i]);
        i64 x, y;
        if (i < 4) {
            const LimbC m1 = fx_limbs(mr[i + 1], mi[i + 1]), v1 = fx_limbs(h.re[i + 1], h.im[i + 1]);
            auto c = [&](i64 a) { return i == 0 || i == 3 ? a : a + fx_mul(r32m1, fx_split(a)); };
            fx_conj_mul(m, v1, x, y);
            const int su = E.G[i] + E.T[i + 1] - E.xy, sd = E.G[i + 1] + E.T[i] - E.xy;
            S.upr += c(fx_scale_any(x, su));
            S.upi += c(fx_scale_any(y, su));
            fx_conj_mul(m1, v, x, y);
            S.dnr += c(fx_scale_any(x, sd));
            S.dni += c(fx_scale_any(y, sd));
        }
        if (i != 2) S.z += (2 - i) * fx_scale_any(fx_conj_mul_im(m, v), E.G[i] + E.T[i] - E.z);
        // conj(p) v - conj(t) mu
        fx_conj_mul(p, v, x, y);
        const int sv = E.dG + E.T[i] - E.q[i], sm = E.dT + E.G[i] - E.q[i];
        S.qr[i] += fx_scale_any(x, sv);
        S.qi[i] += fx_scale_any(y, sv);
        fx_conj_mul(t, m, x, y);
        S.qr[i] -= fx_scale_any(x, sm);
        S.qi[i] -= fx_scale_any(y, sm);
    }
    S.s += fx_conj_mul_im(p, t);
}

// The FP32 steps: an iterate kept for the reverse sweep with its dot product, and the sums in units of 2^exponent
struct FxSlotF {
    FxCpxF v[5], dot;
};
struct FxSumsF {
    FxCpxF up, dn, q[5];
    float z, s;
};
__device__ __forceinline__ FxCpxF fx_conj_mac(FxCpxF a, FxCpxF b, FxCpxF acc) {
    return {fmaf(a.re, b.re, fmaf(a.im, b.im, acc.re)), fmaf(a.re, b.im, fmaf(-a.im, b.re, acc.im))};
}
__device__ __forceinline__ FxCpxF operator*(float c, FxCpxF a) { return {c * a.re, c * a.im}; }

// v_k from x: the Horner steps K .. k + 1
__device__ __noinline__ void fx_horner_again(const FxWF* W, const FxCpxF* x, int K, int k, FxSlotF* out) {
    FxCpxF v[5], o[5];
    for (int i = 0; i < 5; ++i) v[i] = x[i];
    for (int n = K; n > k; --n) {
        fx_apply_f(*W, v, fx_dot_f(*W, v), o, fx_inv(n));
        for (int i = 0; i < 5; ++i) v[i] = {x[i].re + o[i].re, x[i].im + o[i].im};
    }
    for (int i = 0; i < 5; ++i) out->v[i] = v[i];
    out->dot = fx_dot_f(*W, v);
}

// Step k of the reverse sweep (ik = 1/k): lam = lambda_{k-1} -> lambda_k, v = v_k
__device__ __forceinline__ void fx_reverse_f(const FxWF& W, const FxAdjExp& E, FxCpxF lam[5], const FxSlotF& h, float ik, FxSumsF& S) {
    FxCpxF mu[5], o[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) mu[i] = ik * lam[i];
    const FxCpxF p = fx_dot_f(W, mu), nt = {-h.dot.re, -h.dot.im};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        if (i < 4) {
            const float c = i == 0 || i == 3 ? 1.f : 1.2247449f;
            S.up = fx_conj_mac((c * fx_pow2f(E.G[i] + E.T[i + 1] - E.xy)) * mu[i], h.v[i + 1], S.up);
            S.dn = fx_conj_mac((c * fx_pow2f(E.G[i + 1] + E.T[i] - E.xy)) * mu[i + 1], h.v[i], S.dn);
        }
        if (i != 2) {
            const FxCpxF m = (float(2 - i) * fx_pow2f(E.G[i] + E.T[i] - E.z)) * mu[i];
            S.z = fmaf(m.re, h.v[i].im, fmaf(-m.im, h.v[i].re, S.z));
        }
        S.q[i] = fx_conj_mac(fx_pow2f(E.dG + E.T[i] - E.q[i]) * p, h.v[i], S.q[i]);
        S.q[i] = fx_conj_mac(fx_pow2f(E.dT + E.G[i] - E.q[i]) * nt, mu[i], S.q[i]);
    }
    S.s = fmaf(p.re, h.dot.im, fmaf(-p.im, h.dot.re, S.s));
    fx_apply_f(W, mu, p, o, 1.f);
#pragma unroll
    for (int i = 0; i < 5; ++i) lam[i] = {-o[i].re, -o[i].im};  // i W mu
}

// v / k
QLGA_HD i64 fx_div(i64 v, Limb ik) { return fx_mul(ik, fx_split(v)); }

// The pull-back at a site of a warp; the arguments are those of potential_vjp_site.  Returns false, with nothing
// changed, outside the domain (that of fx_unitary, also for the cotangents, and those below 2^400).  All 32 lanes take part.
__device__ __forceinline__ bool fx_vjp_site(const cpx<double> a[5], const cpx<double> b[5], cpx<double> ga[5],
                                            cpx<double> gb[5], const AdjConst<double>& A, double dc[3]) {
    const FixPot& C = A.pc.fx;
    bool ok = true;
    i64 xr[5], xi[5], yr[5], yi[5], gr[5], gi[5], hr[5], hi[5];  // a + b, a - b, ga + gb, ga - gb
    FxLevels psi;
    FxSizes z;
    FxAdjExp E;
    FxForms f;
    float w;
    {
        float Lx[5], Lg[5];
        int ex[5], eg[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const unsigned mx = fx_top(fx_top(fx_top(fx_top(0, a[i].re), a[i].im), b[i].re), b[i].im);
            const unsigned mg = fx_top(fx_top(fx_top(fx_top(0, ga[i].re), ga[i].im), gb[i].re), gb[i].im);
            const int Ex = fx_level_exponent(mx, ok), Eg = fx_exponent(mg);
            ok = ok && mg < (unsigned(1023 + 400) << 20) && (mg == 0 || mg >= (unsigned(kFxMinExp + 1) << 20));
            ex[i] = Ex - 1022 - 60;
            eg[i] = Eg - 1022 - 60;
            const i64 a0 = fx_from_double<60>(a[i].re, Ex), a1 = fx_from_double<60>(a[i].im, Ex);
            const i64 b0 = fx_from_double<60>(b[i].re, Ex), b1 = fx_from_double<60>(b[i].im, Ex);
            const i64 c0 = fx_from_double<60>(ga[i].re, Eg), c1 = fx_from_double<60>(ga[i].im, Eg);
            const i64 d0 = fx_from_double<60>(gb[i].re, Eg), d1 = fx_from_double<60>(gb[i].im, Eg);
            xr[i] = a0 + b0;
            xi[i] = a1 + b1;
            yr[i] = a0 - b0;
            yi[i] = a1 - b1;
            gr[i] = c0 + d0;
            gi[i] = c1 + d1;
            hr[i] = c0 - d0;
            hi[i] = c1 - d1;
            fx_level(xr[i], xi[i], ex[i], psi.p.re[i], psi.p.im[i], psi.e[i]);
            z.p[i] = fx_log_of(xr[i], xi[i], ex[i]);
            Lx[i] = fmaxf(fmaxf(z.p[i], fx_log_of(yr[i], yi[i], ex[i])), float(kFxFloor));
            Lg[i] = fmaxf(fmaxf(fx_log_of(gr[i], gi[i], eg[i]), fx_log_of(hr[i], hi[i], eg[i])), float(kFxFloor));
        }
        fx_forms(psi, C, f);
        z.e = fx_log_of(f.er, f.ei, f.ee - 60);
        z.R = C.R_log;
        w = fmaxf(fx_exponents(z, f, C, Lx, E.T), fx_exponents(z, f, C, Lg, E.G));
        ok = ok && w <= kFxNormMax;
        if (!fx_warp_all(ok)) return false;
        E.dT = fx_dot_exp(psi.e, E.T);
        E.dG = fx_dot_exp(psi.e, E.G);
        E.sums();
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const int nx = fx_clamp(ex[i] + 56 - E.T[i], -63, 57), ng = fx_clamp(eg[i] + 57 - E.G[i], -63, 57);
            xr[i] = fx_scale(xr[i], nx);
            xi[i] = fx_scale(xi[i], nx);
            yr[i] = fx_scale(yr[i], nx);
            yi[i] = fx_scale(yi[i], nx);
            gr[i] = fx_scale(gr[i], ng);
            gi[i] = fx_scale(gi[i], ng);
            hr[i] = fx_scale(hr[i], ng);
            hi[i] = fx_scale(hi[i], ng);
        }
    }
    const float wmax = fx_warp_max(w);
    const int K = fx_degree(wmax, kFxTol);
    const int kA = max(1, min(K, fx_degree(wmax, kFxTolF) + 1));  // w^kA / kA! <= 2^-31
    FxW WT, WG;
    fx_build_w(psi, f, C, E.T, WT);
    fx_build_w(psi, f, C, E.G, WG);
    i64 pc, ps;
    fx_site_phase(f.rho, f.en - 56, C, pc, ps);

    FxAdjSums S;
    S.upr = S.upi = S.dnr = S.dni = S.z = S.s = S.tau = 0;
    FxSumsF F;
    F.up = F.dn = {0.f, 0.f};
    F.z = F.s = 0.f;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        S.qr[i] = S.qi[i] = 0;
        F.q[i] = {0.f, 0.f};
    }
    const float s56 = 1.3877788e-17f, s57 = 6.9388939e-18f;  // 2^-56, 2^-57
    auto op_f = [](i64 v, float c) { return fx_float(fx_split(v), c); };
    FxAdjSlot kept[kFxAdjSlots];
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {  // one copy of the code for both vectors
        fx_rotate(pc, -ps, gr, gi);  // lambda_0 = e^{i theta} g
        // forward sweep
        i64 vr[5], vi[5];
        FxCpxF xf[5];
        FxSlotF keptf[kAdjSlotsF];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            vr[i] = xr[i];
            vi[i] = xi[i];
        }
        if (K > kA) {  // warp-uniform
            const FxWF Wf(WT);
            FxSlotF h;
            FxCpxF o[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) h.v[i] = xf[i] = {op_f(xr[i], s56), op_f(xi[i], s56)};
#pragma unroll 1
            for (int k = K;; --k) {
                h.dot = fx_dot_f(Wf, h.v);
                if (k - kA <= kAdjSlotsF) keptf[k - kA - 1] = h;
                fx_apply_f(Wf, h.v, h.dot, o, fx_inv(k));
                if (k == kA + 1) {
                    auto whole = [](float x) {  // |x| < 2^57
                        const int top = fx_rint(x * 1.4901161e-8f);  // 2^-26
                        return (i64(top) << 26) + fx_rint(fmaf(float(top), -67108864.f, x));
                    };
                    const float one = 72057594037927936.f;  // 2^56
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        vr[i] += whole(o[i].re * one);
                        vi[i] += whole(o[i].im * one);
                    }
                    break;
                }
#pragma unroll
                for (int i = 0; i < 5; ++i) h.v[i] = {xf[i].re + o[i].re, xf[i].im + o[i].im};
            }
        }
#pragma unroll 1
        for (int k = kA; k >= 1; --k) {
            FxAdjSlot& h = kept[k - 1];
            i64 wr[5], wi[5];
            fx_apply_ints(WT, vr, vi, wr, wi);
            const Limb ik = {c_fx_inv_int.h[k], c_fx_inv_int.l[k]};
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                h.re[i] = vr[i];
                h.im[i] = vi[i];
                vr[i] = xr[i] + fx_div(wr[i], ik);
                vi[i] = xi[i] + fx_div(wi[i], ik);
            }
        }
#pragma unroll
        for (int i = 0; i < 5; ++i)  // tau += Im lambda_0^dagger v_0
            S.tau += fx_scale_any(fx_conj_mul_im(fx_limbs(gr[i], gi[i]), fx_limbs(vr[i], vi[i])), E.G[i] + E.T[i] - E.tau);
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
            fx_apply_ints(WG, lr, li, wr, wi);
            fx_contract(S, E, WT, WG, lr, li, kept[k - 1]);
#pragma unroll
            for (int i = 0; i < 5; ++i) {  // lambda_k = i W mu = -(-i W mu)
                lr[i] = -wr[i];
                li[i] = -wi[i];
                gr[i] += lr[i];
                gi[i] += li[i];
            }
        }
        if (K > kA) {
            const FxWF Wf(WG);
            FxCpxF lf[5], sf[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                lf[i] = {op_f(lr[i], s57), op_f(li[i], s57)};
                sf[i] = {0.f, 0.f};
            }
#pragma unroll 1
            for (int k = kA + 1; k <= K; ++k) {
                FxSlotF h;
                if (k - kA <= kAdjSlotsF) {
                    h = keptf[k - kA - 1];
                } else {
                    const FxWF Wc(WT);
                    FxCpxF xc[5];
                    FxSlotF hc;
                    for (int i = 0; i < 5; ++i) xc[i] = xf[i];
                    fx_horner_again(&Wc, xc, K, k, &hc);
                    h = hc;
                }
                fx_reverse_f(Wf, E, lf, h, fx_inv(k), F);
#pragma unroll
                for (int i = 0; i < 5; ++i) sf[i] = {sf[i].re + lf[i].re, sf[i].im + lf[i].im};
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
    // The sums are of psi with ga + gb and of d with ga - gb: twice those of a with ga and b with gb.
    auto join = [](i64 v, float x, int e) { return fma(double(x), fx_pow2_or_0(e - 1), double(v) * fx_pow2_or_0(e - 54)); };
    const double upr = join(S.upr, F.up.re, E.xy), upi = join(S.upi, F.up.im, E.xy);
    const double dnr = join(S.dnr, F.dn.re, E.xy), dni = join(S.dni, F.dn.im, E.xy);
    const double phx = upi + dni, phy = dnr - upr, phz = join(S.z, F.z, E.z);
    const double tau = join(S.tau, 0.f, E.tau);
    cpx<double> psid[5], h[5];
    const double t0 = 2.0 * A.dg0 * tau, t1 = 2.0 * A.dg1;
    const cpx<double> lower = {t1 * phx, t1 * phy};
#pragma unroll
    for (int i = 0; i < 5; ++i) psid[i] = a[i] + b[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const double sg = (i & 1) ? -A.dg2_5 : A.dg2_5;
        const double qr = join(S.qr[4 - i], F.q[4 - i].re, E.q[4 - i]), qi = join(S.qi[4 - i], F.q[4 - i].im, E.q[4 - i]);
        h[i] = fma(double(2 - i), t1 * phz, t0) * psid[i];
        h[i] = {fma(sg, qi, h[i].re), fma(sg, qr, h[i].im)};  // i conj(q)
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const cpx<double> l = spin_c<double>(i) * lower;
        h[i] = cfmac(l, psid[i + 1], h[i]);
        h[i + 1] = cfma(l, psid[i], h[i + 1]);
    }
    const double un = fx_pow2_or_0(f.en - 56), uf = fx_pow2_or_0(f.fe - 55);
    dc[0] = A.delta * (double(f.rho) * un) * tau;
    dc[1] = A.delta * ((double(f.fr) * uf) * phx + (double(f.fi) * uf) * phy + (double(f.Fz) * un) * phz);
    dc[2] = A.delta * join(S.s, F.s, E.dT + E.dG) / 5.0;
    // U^dagger of the cotangents: half the sum and the difference
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const FxToDouble to(E.G[i] - 58);
        ga[i] = {to(gr[i] + hr[i]) + h[i].re, to(gi[i] + hi[i]) + h[i].im};
        gb[i] = {to(gr[i] - hr[i]) + h[i].re, to(gi[i] - hi[i]) + h[i].im};
    }
    return true;
}

}  // namespace qlga
