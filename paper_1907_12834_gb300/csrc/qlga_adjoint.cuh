// qlga_adjoint.cuh -- reverse mode (adjoint) of the plain QLGA step (arXiv:1907.12834, Sec. VII.B).
//
// For a real loss L of the state, the cotangent of a complex amplitude z is gbar = dL/dRe z +
// i dL/dIm z (so dL = Re sum conj(gbar) dz); a cotangent buffer has the state's layout.  One
// plain step x' = K U(x) x pulls a cotangent back as
//   gbar_x = U_x^T (K^dagger gbar_x')
// where K^dagger is the adjoint kinetic operator (axes, blocks and factors in reverse order, each
// factor replaced by its adjoint) and U_x^T the transposed linearisation of the potential step at
// the state x, which includes the dependence of V on psi.
//
// Potential step at one site (a' = U a, b' = U b, U = exp(-i delta V(psi)), psi = a + b):
//   gbar_a = U^dagger gbar_a' + h,   gbar_b = U^dagger gbar_b' + h,
// with h the gradient through psi.  Writing V = c 1 + W (c = (g0 + g2/10) rho) and B = -i delta W,
// U = e^{-i delta c} P(B) with P the degree-K Taylor polynomial of the forward step in Horner form,
//   v_K = x,  v_{k-1} = x + B v_k / k,  P x = v_0.
// Its reverse sweep starts from lambda_0 = e^{i delta c} gbar' and runs upwards,
//   mu_k = lambda_{k-1} / k,  lambda_k = B^dagger mu_k,  P^dagger lambda_0 = sum_k lambda_k,
// and step k adds Im mu_k^dagger d(delta W) v_k to dL.  Summed over the steps and over x = a, b,
//   phi_nu = Im sum mu_k^dagger f_nu v_k                                            (nu = x, y, z)
//   q      = sum conj(u . mu_k) v_k - conj(u . v_k) mu_k,  u_m = (-1)^m psi_{-m} = conj(s_m)
//   tau    = Im lambda_0^dagger P x
//   h      = delta [2 g0 tau psi + 2 g1 sum_nu phi_nu f_nu psi + (g2/5) i J conj(q)]
// and the coupling gradients are dL/dg0 = delta rho tau, dL/dg1 = delta sum_nu F_nu phi_nu,
// dL/dg2 = (delta/5) Im sum conj(u . mu_k) (u . v_k).  (The identity direction of dV commutes with B; its
// derivative uses the exact exponential, whose trace form is tau.)
//
// Two applications of W per Taylor term and vector, four in all, where the Frechet derivatives of
// the same polynomial by augmented Horner recursions, one per spin direction and two for the singlet
// term, took fourteen (a gradient of 24 steps on 512^2 in FP32 4.03 -> 3.56 ms, of 12 on 256^2 in FP64
// 17.1 -> 9.4 ms).  The Horner iterates wait for the reverse sweep in thread-local memory.
#pragma once

#include "qlga_device.cuh"

namespace qlga {

// ------------------------------------------------------------------ adjoint kinetic stencil
//
// K^dagger of one axis: the blocks' adjoints in reverse order.  A block I'_c = S_c C' S^T_c C has
// adjoint C^dagger S_c C'^dagger S^T_c (S^T_c acts first).  In the (a, bt) basis the real parts
// of the collides' adjoints are [[1, -1], [1, 1]] (adjoint of [[1, 1], [-1, 1]]) and vice versa;
// their scalar prefactors multiply to exactly 1/16 per axis, as for K.  Derived at compile time
// from the block definition on a unit impulse, like the forward table.
constexpr KinStencil make_stencil_adjoint(int variant) {
    KinStencil S{};
    const int block_qubit_rev[4] = {0, 0, 1, 1};
    for (int src = 0; src < 2; ++src) {
        int v[2][11] = {};
        v[src][5] = 1;
        for (int blk = 0; blk < 4; ++blk) {
            const int c = block_qubit_rev[blk];
            shift_int(v, c, -1);          // (S_c)^dagger = S^T_c
            collide_int(v, 1, -1, 1, 1);  // C'^dagger (C' is [[1, 1], [-1, 1]] in both variants)
            shift_int(v, c, +1);          // (S^T_c)^dagger = S_c
            if (variant == 0) collide_int(v, 1, -1, 1, 1);  // C^dagger, K1
            else collide_int(v, 1, 1, -1, 1);               // C^dagger, K2
        }
        for (int dst = 0; dst < 2; ++dst)
            for (int k = -4; k <= 4; ++k) S.g[dst][src][k + 4] = v[dst][5 - k];
    }
    return S;
}

constexpr KinStencil kStencilAdj[2] = {make_stencil_adjoint(0), make_stencil_adjoint(1)};

// ------------------------------------------------------------------ per-site pull-back of U

template <class T>
struct AdjConst {
    PotConst<T> pc;  // the forward step's constants (delta folded in)
    T dg0;           // delta g0
    T dg1;           // delta g1
    T dg2_5;         // delta g2 / 5
    T delta;
    AdjConst() = default;
    __host__ explicit AdjConst(const PotParams& P)
        : pc(P), dg0(T(P.delta * P.g0)), dg1(T(P.delta * P.g1)), dg2_5(T(P.delta * P.g2 / 5.0)),
          delta(T(P.delta)) {}
};

// Spin matrices of Sec. II on a 5-vector (rows m = +2..-2): off-diagonal entries c_i of f_x at
// (i, i+1) and (i+1, i); f_y has -i c_i and +i c_i there; f_z = diag(2, 1, 0, -1, -2).
template <class T>
__device__ __forceinline__ T spin_c(int i) {
    return (i == 0 || i == 3) ? T(1) : T(1.2247448713915890491);  // 1, sqrt(3/2), sqrt(3/2), 1
}

// conj(x) . y
template <class T>
__device__ __forceinline__ cpx<T> cdot(const cpx<T> x[5], const cpx<T> y[5]) {
    cpx<T> acc = cmulc(x[0], y[0]);
#pragma unroll
    for (int i = 1; i < 5; ++i) acc = cfmac(x[i], y[i], acc);
    return acc;
}

// v = x - i ik w   (one Horner step of P(B) with B v = -i W v)
template <class T>
__device__ __forceinline__ void horner_down(const cpx<T> x[5], const cpx<T> w[5], cpx<T> v[5], T ik) {
#pragma unroll
    for (int i = 0; i < 5; ++i) v[i] = {fma(ik, w[i].im, x[i].re), fma(-ik, w[i].re, x[i].im)};
}

// The forward step's W at a site (as potential_site builds it, unscaled input) and its degree.
template <class T>
__device__ __forceinline__ int build_w(const cpx<T> psi[5], const PotConst<T>& C, WOp<T>& W, T& rho,
                                       T& Fz, cpx<T>& Fp, unsigned* status, T* beta_out = nullptr) {
    T n[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) n[i] = norm2(psi[i]);
    rho = (n[0] + n[1]) + (n[2] + n[3]) + n[4];
    Fz = T(2) * (n[0] - n[4]) + (n[1] - n[3]);
    const T r32 = T(1.2247448713915890491);
    Fp = cmulc(psi[0], psi[1]);
    Fp = cfmac(psi[3], psi[4], Fp);
    cpx<T> mid = cmulc(psi[1], psi[2]);
    mid = cfmac(psi[2], psi[3], mid);
    Fp = {fma(r32, mid.re, Fp.re), fma(r32, mid.im, Fp.im)};
    Fp = T(2) * Fp;
    const T Fabs = sqrt(fma(Fz, Fz, norm2(Fp)));
    const T beta = fma(C.b1, Fabs, C.b2 * rho);
    if (!(beta <= T(kBetaMax))) atomicOr(status, 1u);
    if (beta_out) *beta_out = beta;
    const int K = warp_taylor_degree(beta, TaylorTol<T>::value);
    const T g2r = C.dr * rho;
    const T gz = C.dz * Fz;
    W.D[0] = T(2) * gz - g2r;
    W.D[1] = gz - g2r;
    W.D[2] = -g2r;
    W.D[3] = -gz - g2r;
    W.D[4] = T(-2) * gz - g2r;
    W.ep[0] = C.e0 * Fp;
    W.ep[1] = C.e1 * Fp;
    W.ep[2] = W.ep[1];
    W.ep[3] = W.ep[0];
    W.u[0] = psi[4];
    W.u[1] = {-psi[3].re, -psi[3].im};
    W.u[2] = psi[2];
    W.u[3] = {-psi[1].re, -psi[1].im};
    W.u[4] = psi[0];
    W.R = C.R;
    return K;
}

// FP64 pull-backs run the steps of order above k0 of both sweeps in FP32 (Kin = K - k0 of them) and
// the k0 others in FP64, as the forward step does (zframe_inner_fp32), with k0 the smallest
// order whose bound beta^k0 / k0! is at most kAdjInnerTol.  The last FP32 step adds its increment to the exact
// x, so v_k0 is good to 2^-24 beta / (k0 + 1); it meets mu_k0, of order beta^(k0 - 1) / k0!, and FP32 sees
// only mu_k of order beta^k0 / (k0 + 1)! and less: 2^-55 of the sums either way.
constexpr double kAdjInnerTol = 4.656612873077393e-10;  // 2^-31

template <class U>
__device__ __forceinline__ cpx<U> to_prec(cpx<double> z) { return {U(z.re), U(z.im)}; }

template <class U>
__device__ __forceinline__ WOp<U> wop_to(const WOp<double>& W) {
    WOp<U> V;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        V.D[i] = U(W.D[i]);
        V.u[i] = to_prec<U>(W.u[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) V.ep[i] = to_prec<U>(W.ep[i]);
    V.R = U(W.R);
    return V;
}

// u . x
template <class U>
__device__ __forceinline__ cpx<U> singlet_dot(const WOp<U>& W, const cpx<U> x[5]) {
    cpx<U> t0 = cmul(W.u[0], x[0]), t1 = cmul(W.u[1], x[1]);
    t0 = cfma(W.u[2], x[2], t0);
    t1 = cfma(W.u[3], x[3], t1);
    return cfma(W.u[4], x[4], t0) + t1;
}
// y = W x with u . x given
template <class U>
__device__ __forceinline__ void apply_dotted(const WOp<U>& W, const cpx<U> x[5], cpx<U> dot, cpx<U> y[5]) {
    const cpx<U> t = W.R * dot;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const cpx<U> tu = cmulc(W.u[i], t);
        y[i] = {fma(W.D[i], x[i].re, tu.re), fma(W.D[i], x[i].im, tu.im)};
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        y[i] = cfmac(W.ep[i], x[i + 1], y[i]);
        y[i + 1] = cfma(W.ep[i], x[i], y[i + 1]);
    }
}

// A Horner iterate kept for the reverse sweep, with u . v
template <class U>
struct HornerSlot {
    cpx<U> v[5], dot;
};
// Iterates kept per thread: k = 1 .. kAdjSlots in the arithmetic of the state, and of an FP64 state's
// FP32 steps the kAdjSlotsF lowest.  Denser sites, whose degree is higher, form the others again.
template <class T>
constexpr int kAdjSlots = std::is_same<T, float>::value ? 4 : 6;
constexpr int kAdjSlotsF = 4;

template <class U>
__device__ __noinline__ void horner_again(const WOp<U>* W, const cpx<U>* x, int K, int k, HornerSlot<U>* out) {
    cpx<U> v[5], w[5];
    for (int i = 0; i < 5; ++i) v[i] = x[i];
    for (int n = K; n > k; --n) {
        W->apply(v, w);
        horner_down(x, w, v, inv_k(n, U(0)));
    }
    for (int i = 0; i < 5; ++i) out->v[i] = v[i];
    out->dot = singlet_dot(*W, v);
}

// Sums of the reverse sweep over the steps and vectors
template <class U>
struct AdjSweep {
    cpx<U> up[2], dn[2];  // conj(mu_i) v_{i+1} and conj(mu_{i+1}) v_i, over c_i = 1 and over c_i = sqrt(3/2)
    U z1, z2;             // Im conj(mu_m) v_m over m = +-1 (signed) and m = +-2
    cpx<U> q[5];
    U s;                  // Im conj(u . mu) (u . v)
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < 2; ++i) up[i] = dn[i] = {U(0), U(0)};
#pragma unroll
        for (int i = 0; i < 5; ++i) q[i] = {U(0), U(0)};
        z1 = z2 = s = U(0);
    }
};

// Step k of the reverse sweep (ik = 1/k): lam = lambda_{k-1} -> lambda_k, v = v_k
template <class U>
__device__ __forceinline__ void reverse_step(const WOp<U>& W, cpx<U> lam[5], const HornerSlot<U>& h, U ik, AdjSweep<U>& S) {
    cpx<U> mu[5], w[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) mu[i] = ik * lam[i];
    const cpx<U> p = singlet_dot(W, mu), nt = {-h.dot.re, -h.dot.im};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = i == 0 || i == 3 ? 0 : 1;
        S.up[c] = cfmac(mu[i], h.v[i + 1], S.up[c]);
        S.dn[c] = cfmac(mu[i + 1], h.v[i], S.dn[c]);
    }
    auto im = [&](int i, U acc) { return fma(mu[i].re, h.v[i].im, fma(-mu[i].im, h.v[i].re, acc)); };
    S.z2 = im(0, S.z2) - im(4, U(0));
    S.z1 = im(1, S.z1) - im(3, U(0));
#pragma unroll
    for (int i = 0; i < 5; ++i) S.q[i] = cfmac(nt, mu[i], cfmac(p, h.v[i], S.q[i]));
    S.s = fma(p.re, h.dot.im, fma(-p.im, h.dot.re, S.s));
    apply_dotted(W, mu, p, w);
#pragma unroll
    for (int i = 0; i < 5; ++i) lam[i] = {-w[i].im, w[i].re};  // B^dagger = i W
}

// Both sweeps of one vector x with its cotangent g = lambda_0: g <- P^dagger g, tau += Im g^dagger P x,
// S += the sums.  Wf: W in FP32, for the Kin inner steps of an FP64 state.
template <class T>
__device__ __forceinline__ void pull_back_vector(const WOp<T>& W, const WOp<float>& Wf, const cpx<T> x[5], cpx<T> g[5],
                                                 int K, int Kin, T& tau, AdjSweep<T>& S) {
    constexpr bool kMixed = std::is_same<T, double>::value;
    HornerSlot<T> kept[kAdjSlots<T>];
    [[maybe_unused]] HornerSlot<float> keptf[kMixed ? kAdjSlotsF : 1];
    [[maybe_unused]] cpx<float> xf[5];
    const int k0 = K - Kin;
    HornerSlot<T> h;
#pragma unroll
    for (int i = 0; i < 5; ++i) h.v[i] = x[i];
    if constexpr (kMixed) {
        if (Kin > 0) {  // warp-uniform
            HornerSlot<float> f;
#pragma unroll
            for (int i = 0; i < 5; ++i) f.v[i] = xf[i] = to_prec<float>(x[i]);
#pragma unroll 1
            for (int k = K;; --k) {
                f.dot = singlet_dot(Wf, f.v);
                if (k - k0 <= kAdjSlotsF) keptf[k - k0 - 1] = f;
                cpx<float> w[5];
                apply_dotted(Wf, f.v, f.dot, w);
                const float ik = inv_k(k, 0.f);
                if (k == k0 + 1) {  // warp-uniform
#pragma unroll
                    for (int i = 0; i < 5; ++i) h.v[i] = {x[i].re + double(ik * w[i].im), x[i].im - double(ik * w[i].re)};
                    break;
                }
                horner_down(xf, w, f.v, ik);
            }
        }
    }
#pragma unroll 1
    for (int k = k0; k >= 1; --k) {
        h.dot = singlet_dot(W, h.v);
        if (k <= kAdjSlots<T>) kept[k - 1] = h;
        cpx<T> w[5];
        apply_dotted(W, h.v, h.dot, w);
        horner_down(x, w, h.v, inv_k(k, T(0)));
    }
    tau += cdot(g, h.v).im;
    cpx<T> lam[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) lam[i] = g[i];
#pragma unroll 1
    for (int k = 1; k <= k0; ++k) {
        if (k <= kAdjSlots<T>) {
            h = kept[k - 1];
        } else {  // the iterates of the dense sites
            WOp<T> Wc = W;
            cpx<T> xc[5];
            HornerSlot<T> hc;
            for (int i = 0; i < 5; ++i) xc[i] = x[i];
            horner_again<T>(&Wc, xc, K, k, &hc);
            h = hc;
        }
        reverse_step(W, lam, h, inv_k(k, T(0)), S);
#pragma unroll
        for (int i = 0; i < 5; ++i) g[i] = g[i] + lam[i];
    }
    if constexpr (kMixed) {
        if (Kin > 0) {
            AdjSweep<float> F;
            F.clear();
            cpx<float> lf[5], gf[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                lf[i] = to_prec<float>(lam[i]);
                gf[i] = {0.f, 0.f};
            }
#pragma unroll 1
            for (int k = k0 + 1; k <= K; ++k) {
                HornerSlot<float> f;
                if (k - k0 <= kAdjSlotsF) {
                    f = keptf[k - k0 - 1];
                } else {
                    WOp<float> Wc = Wf;
                    cpx<float> xc[5];
                    HornerSlot<float> fc;
                    for (int i = 0; i < 5; ++i) xc[i] = xf[i];
                    horner_again<float>(&Wc, xc, K, k, &fc);
                    f = fc;
                }
                reverse_step(Wf, lf, f, inv_k(k, 0.f), F);
#pragma unroll
                for (int i = 0; i < 5; ++i) gf[i] = gf[i] + lf[i];
            }
            auto add = [](cpx<double>& d, cpx<float> v) { d = {d.re + double(v.re), d.im + double(v.im)}; };
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                add(g[i], gf[i]);
                add(S.q[i], F.q[i]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                add(S.up[i], F.up[i]);
                add(S.dn[i], F.dn[i]);
            }
            S.z1 += double(F.z1);
            S.z2 += double(F.z2);
            S.s += double(F.s);
        }
    }
}

// Pull-back through U at one site.  (a, b): the state before U.  (ga, gb): cotangents of the
// outputs on entry, of the inputs on exit.  dc[3] = this site's dL/d(g0, g1, g2).
template <class T>
__device__ __forceinline__ void potential_vjp_site(const cpx<T> a[5], const cpx<T> b[5], cpx<T> ga[5],
                                                   cpx<T> gb[5], const AdjConst<T>& A, T dc[3],
                                                   unsigned* status) {
    cpx<T> psi[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) psi[i] = a[i] + b[i];
    WOp<T> W;
    T rho, Fz, beta;
    cpx<T> Fp;
    const int K = build_w(psi, A.pc, W, rho, Fz, Fp, status, &beta);
    int Kin = 0;  // FP64: inner Horner steps in FP32 (kAdjInnerTol)
    WOp<float> Wf;
    if constexpr (std::is_same<T, double>::value) {
        const int k0 = warp_max_int(taylor_degree(beta, kAdjInnerTol) + 1);
        Kin = K > k0 ? K - k0 : 0;
        Wf = wop_to<float>(W);
    }
    T sn, cs;
    sin_cos(A.pc.cphase * rho, &sn, &cs);
    const cpx<T> phc = {cs, sn};  // e^{i delta c}
    AdjSweep<T> S;
    S.clear();
    T tau = T(0);
    cpx<T> x[5], y[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        x[i] = a[i];
        y[i] = b[i];
        ga[i] = cmul(phc, ga[i]);
        gb[i] = cmul(phc, gb[i]);
    }
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {  // one copy of the code for both vectors
        pull_back_vector(W, Wf, x, ga, K, Kin, tau, S);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            x[i] = y[i];
            const cpx<T> t = ga[i];
            ga[i] = gb[i];
            gb[i] = t;
        }
    }
    const T r32 = T(1.2247448713915890491);  // sqrt(3/2)
    const cpx<T> up = S.up[0] + r32 * S.up[1], dn = S.dn[0] + r32 * S.dn[1];
    const T phx = up.im + dn.im, phy = dn.re - up.re, phz = fma(T(2), S.z2, S.z1);

    // h = 2 dg0 tau psi + 2 dg1 (phi_z f_z + phi_x f_x + phi_y f_y) psi + dg2/5 i J conj(q)
    const T t0 = T(2) * A.dg0 * tau, t1 = T(2) * A.dg1;
    const cpx<T> lower = {t1 * phx, t1 * phy};  // entry (i + 1, i) per c_i; (i, i + 1) its conjugate
    cpx<T> h[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const T sg = (i & 1) ? -A.dg2_5 : A.dg2_5;
        h[i] = fma(T(2 - i), t1 * phz, t0) * psi[i];
        h[i] = {fma(sg, S.q[4 - i].im, h[i].re), fma(sg, S.q[4 - i].re, h[i].im)};  // i conj(q)
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const cpx<T> l = spin_c<T>(i) * lower;
        h[i] = cfmac(l, psi[i + 1], h[i]);
        h[i + 1] = cfma(l, psi[i], h[i + 1]);
    }

    // coupling gradients
    dc[0] = A.delta * rho * tau;
    dc[1] = A.delta * (Fp.re * phx + Fp.im * phy + Fz * phz);
    dc[2] = A.delta * S.s / T(5);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        ga[i] = ga[i] + h[i];
        gb[i] = gb[i] + h[i];
    }
}

}  // namespace qlga
