// qlga_step1d_f64.cuh -- the fused 1D FP64 step in integer fixed point.
//
// GB300 issues one FP64 instruction per SM sub-partition every 64-76 cycles (qlga_fixed.cuh); the nine-point
// stencil of K alone is 240 of them a site, 16 k cycles of a warp, longer than all of U on integers.
// K's taps are small integers, so here K runs on integers too, exactly up to the conversion of its
// inputs and one rounding of its sum, and feeds U (fx_unitary) without a conversion in between.
// 32768 sites (two solitons): 13 us a step.  Of 100 steps with load and read-out, 16384 sites took 4.14 ms
// in FP64 and 1.45 ms here, 1.15 ms with five lanes per site (below); 1024 sites 1.67 ms, 0.68 ms with ten.
//
// One warp per CTA, one site per lane: small lattices are bound by the latency of one warp's chain,
// so the warps go one to a sub-partition.  A warp loads its 32 columns and the 4-column periodic halo
// on each side (a lane its own column and five values of the halo), converts them and exchanges them
// through shared memory.
//
// Numbers.  Where the exponents of the 40 columns lie within 2^7 of one another (a soliton of the
// lattice scaling spans 2^6 there) all are converted with the largest: components below 2^58, so
// that the stencil's sums (taps of at most 30 in magnitude) fit.  Otherwise (the edge of a tail,
// empty sites) every column has its own exponent and a lane shifts its nine columns to the largest of
// them.  Either way the resolution is at least 2^-51 of the largest component among the nine columns,
// where FP64 rounds each of the 24 sums at 2^-53.  A warp with a value that is not finite, or outside
// U's domain, takes the FP64 code for both K and U.
#pragma once

#include <cuda_runtime.h>

#include "qlga_batch1d.cuh"
#include "qlga_device.cuh"
#include "qlga_step2d_f64.cuh"  // stencil_tap_int

namespace qlga {

constexpr int kFx1dCols = 40;   // columns a warp reads: 32 and the halo
constexpr int kFx1dSpread = 7;  // exponents within this of the largest share it

// K (and U) of site j in FP64, for the warps that the integer form leaves; all lanes take part.
template <int VARIANT, bool POT>
__device__ __noinline__ void step1d_site_f64(const double* in, double* out, int L, int j, bool store,
                                             const PotConstBase<double>* C, unsigned* status, bool abi = false) {
    cpx<double> a[5], b[5];
#pragma unroll 1
    for (int m = 0; m < 5; ++m) {
        cpx<double> xa = {0.0, 0.0}, xbt = {0.0, 0.0};
        static_for<9>([&](auto kc) {
            constexpr int kk = decltype(kc)::value;
            int jj = (j - 4 + kk) % L;
            jj = jj < 0 ? jj + L : jj;
            const Pair4<double> p = load_raw_pair(in, int64_t(m) * L + jj);
            kin_tap_pq<VARIANT, kk>(cpx<double>{p.v[0], p.v[1]}, cpx<double>{p.v[2], p.v[3]}, xa, xbt);
        });
        if (POT) {
            a[m] = xa;
            b[m] = {xbt.im, -xbt.re};
        } else if (store) {
            const double s = 1.0 / 16.0;
            read_out_pair(xbt, abi);
            store_raw_pair(out, int64_t(m) * L + j, s * xa.re, s * xa.im, s * xbt.re, s * xbt.im);
        }
    }
    if (POT) {
        potential_direct_f64(a, b, C, 1.0 / 256.0, 0.5 / 16.0, status);
        if (store)
            for (int m = 0; m < 5; ++m) store_raw_pq(out, int64_t(m) * L + j, a[m], b[m]);
    }
}

// One fused step (K, then U) of a periodic 1D lattice of L sites held pending K as (P, Q), or K alone
// (POT = false: the true state in the resident layout (a, bt) or, with abi, the ABI's (a, b)).
template <int VARIANT, bool POT>
__global__ void __launch_bounds__(32) k_step1d_f64(const double* __restrict__ in, double* __restrict__ out, int L,
                                                   const __grid_constant__ PotConst<double> C, unsigned* status,
                                                   bool abi) {
    __shared__ longlong2 sp[5][kFx1dCols], sq[5][kFx1dCols];
    __shared__ int se[kFx1dCols];
    const int lane = threadIdx.x;
    const int x0 = int(blockIdx.x) * 32;
    const int j = x0 + lane < L ? x0 + lane : L - 1;  // lanes past the end work on some column and store nothing
    const bool store = x0 + lane < L;
    auto wrap = [&](int x) {
        x %= L;
        return x < 0 ? x + L : x;
    };
    const int hc = 32 + (lane >> 2), hk = lane & 3;  // the lane's halo column and component
    double2 own[10];
    double halo[5];
    {
        const int xo = wrap(x0 - 4 + lane), xh = wrap(x0 - 4 + hc);
        const double2* src = reinterpret_cast<const double2*>(in);
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            own[2 * m] = __ldg(src + 2 * (int64_t(m) * L + xo));
            own[2 * m + 1] = __ldg(src + 2 * (int64_t(m) * L + xo) + 1);
            halo[m] = __ldg(in + 4 * (int64_t(m) * L + xh) + hk);
        }
    }
    unsigned to = 0, th = 0;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
            to = max(to, max(fx_hi(own[2 * m + q].x) & 0x7fffffffu, fx_hi(own[2 * m + q].y) & 0x7fffffffu));
        th = max(th, fx_hi(halo[m]) & 0x7fffffffu);
    }
    th = max(th, __shfl_xor_sync(0xffffffffu, th, 1));
    th = max(th, __shfl_xor_sync(0xffffffffu, th, 2));
    const unsigned top = __reduce_max_sync(0xffffffffu, max(to, th));
    if (top >= (unsigned(1023 + 50) << 20)) {  // warp-uniform; far outside U's domain, or not finite
        const PotConstBase<double> base = C;
        step1d_site_f64<VARIANT, POT>(in, out, L, j, store, &base, status, abi);
        return;
    }
    int Eo = fx_exponent(to), Eh = fx_exponent(th);
    int E = fx_exponent(top);
    // columns without a value take part in no comparison
    const int low = __reduce_min_sync(0xffffffffu, min(Eo == kFxMinExp ? E : Eo, Eh == kFxMinExp ? E : Eh));
    const bool shared = E - low <= kFx1dSpread;
    if (shared) Eo = Eh = E;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        sp[m][lane] = make_longlong2(fx_from_double<58>(own[2 * m].x, Eo), fx_from_double<58>(own[2 * m].y, Eo));
        sq[m][lane] = make_longlong2(fx_from_double<58>(own[2 * m + 1].x, Eo), fx_from_double<58>(own[2 * m + 1].y, Eo));
        longlong2* h = hk < 2 ? &sp[m][hc] : &sq[m][hc];
        reinterpret_cast<i64*>(h)[hk & 1] = fx_from_double<58>(halo[m], Eh);
    }
    if (!shared) {
        se[lane] = Eo;
        if (hk == 0) se[hc] = Eh;
    }
    __syncwarp();

    i64 pr[5], pi[5], dr[5], di[5];
    // sum: the lane's (a, bt) of level m, 16 times the true value, in units of 2^(E - 1022 - 58)
    auto take = [&](int m, cpi xa, cpi xbt) {
        if (POT) {  // to 2^3 units: psi = a - i bt and d = a + i bt below 2^62
            xa = {(xa.re + 4) >> 3, (xa.im + 4) >> 3};
            xbt = {(xbt.re + 4) >> 3, (xbt.im + 4) >> 3};
            pr[m] = xa.re + xbt.im;
            pi[m] = xa.im - xbt.re;
            dr[m] = xa.re - xbt.im;
            di[m] = xa.im + xbt.re;
        } else {
            pr[m] = xa.re;
            pi[m] = xa.im;
            dr[m] = abi ? xbt.im : xbt.re;
            di[m] = abi ? -xbt.re : xbt.im;
        }
    };
    if (shared) {
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            cpi xa = {0, 0}, xbt = {0, 0};
            static_for<9>([&](auto kc) {
                constexpr int kk = decltype(kc)::value;
                stencil_tap_int<VARIANT, kk>(sp[m][lane + kk], sq[m][lane + kk], xa, xbt);
            });
            take(m, xa, xbt);
        }
    } else {
        int sh[9];
        E = kFxMinExp;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            sh[k] = se[lane + k];
            E = max(E, sh[k]);
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) sh[k] = min(E - sh[k], 63);
        auto down = [](longlong2 v, int n) {
            return make_longlong2((((v.x << 1) >> n) + 1) >> 1, (((v.y << 1) >> n) + 1) >> 1);
        };
#pragma unroll 1
        for (int m = 0; m < 5; ++m) {
            cpi xa = {0, 0}, xbt = {0, 0};
            static_for<9>([&](auto kc) {
                constexpr int kk = decltype(kc)::value;
                stencil_tap_int<VARIANT, kk>(down(sp[m][lane + kk], sh[kk]), down(sq[m][lane + kk], sh[kk]), xa, xbt);
            });
            // m is a run-time value here: the results go through the lane's own row of sp and sq
            // once its neighbours have read it
            __syncwarp();
            sp[m][lane] = make_longlong2(xa.re, xa.im);
            sq[m][lane] = make_longlong2(xbt.re, xbt.im);
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const longlong2 p = sp[m][lane], q = sq[m][lane];
            take(m, cpi{p.x, p.y}, cpi{q.x, q.y});
        }
    }

    if (POT) {
        int e = E - 1022 - 55;
        if (!fx_unitary(pr, pi, dr, di, e, -4, true, C.fx)) {
            const PotConstBase<double> base = C;
            step1d_site_f64<VARIANT, POT>(in, out, L, j, store, &base, status, abi);
            return;
        }
        if (!store) return;
        e -= 5;  // 0.5 / 16
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const i64 a0 = pr[m] + dr[m], a1 = pi[m] + di[m], b0 = pr[m] - dr[m], b1 = pi[m] - di[m];
            store_raw_pair(out, int64_t(m) * L + j, fx_pack(a0 - b1, e), fx_pack(a1 + b0, e), fx_pack(a0 + b1, e),
                           fx_pack(a1 - b0, e));
        }
    } else if (store) {
        const int e = E - 1022 - 58 - 4;
#pragma unroll
        for (int m = 0; m < 5; ++m)
            store_raw_pair(out, int64_t(m) * L + j, fx_pack(pr[m], e), fx_pack(pi[m], e), fx_pack(dr[m], e), fx_pack(di[m], e));
    }
}

// ------------------------------------------------------------------ five or ten lanes per site
//
// Lattices too small to fill the GPU with one site per lane: a site's levels sit on five lanes (LPS = 5, six
// sites per warp, each lane both vectors of U) or on ten (LPS = 10, three sites, psi and d = a - b on
// five lanes each), as in qlga_lanes1d.cuh; lanes 30 and 31 repeat lanes 0 and 1 of the last site and
// store nothing.  A warp's chain is then a third as long, and its code a third of the size (one warp per
// sub-partition waits for instructions half of its time on the code of the one-lane form).
// us a step with 10 / 5 / 1 lanes: 1024 sites 4.7 / 6.0 / 11.4, 16384 13.0 / 9.9 / 12.1, 65536 43 / 25 / 19.

__device__ __forceinline__ Limb fx_shfl(Limb v, int src) {
    return {__shfl_sync(0xffffffffu, v.h, src), __shfl_sync(0xffffffffu, v.l, src)};
}

// The lane's place in its group of five, and the group's sums (exact on integers in any order)
struct FxGroup {
    int m, base, s1, s2, s4;
    __device__ __forceinline__ FxGroup(int m_, int base_)
        : m(m_), base(base_), s1(base_ + (m_ + 1) % 5), s2(base_ + (m_ + 2) % 5), s4(base_ + (m_ + 4) % 5) {}
    template <class T>
    __device__ __forceinline__ T sum(T v) const {
        T s = v + __shfl_sync(0xffffffffu, v, s1);
        s += __shfl_sync(0xffffffffu, s, s2);
        return s + __shfl_sync(0xffffffffu, v, s4);
    }
    __device__ __forceinline__ int max_of(int v) const {
        const int s = max(v, __shfl_sync(0xffffffffu, v, s1));
        return max(max(s, __shfl_sync(0xffffffffu, s, s2)), __shfl_sync(0xffffffffu, v, s4));
    }
    __device__ __forceinline__ int up() const { return base + (m < 4 ? m + 1 : 4); }
    __device__ __forceinline__ int down() const { return base + (m > 0 ? m - 1 : 0); }
};

// Bits of the larger of two integers' magnitudes (one's complement)
__device__ __forceinline__ int fx_bits_of(i64 a, i64 b) {
    return 64 - __clzll((a ^ (a >> 63)) | (b ^ (b >> 63)));
}

// The lane's level of K at site j with the exponent of the site's own nine columns (returned), for the
// warps whose columns have no common one.
template <int VARIANT>
__device__ __noinline__ int fx_lane_kinetic_wide(const double* in, int L, int j, FxGroup g, cpi* xa, cpi* xbt) {
    Pair4<double> v[9];
    unsigned top = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        int jj = (j - 4 + k) % L;
        jj = jj < 0 ? jj + L : jj;
        v[k] = load_raw_pair(in, int64_t(g.m) * L + jj);
#pragma unroll
        for (int q = 0; q < 4; ++q) top = max(top, fx_hi(v[k].v[q]) & 0x7fffffffu);
    }
    const int E = fx_exponent(unsigned(g.max_of(int(top))));
    cpi a = {0, 0}, b = {0, 0};
    static_for<9>([&](auto kc) {
        constexpr int kk = decltype(kc)::value;
        stencil_tap_int<VARIANT, kk>(make_longlong2(fx_from_double<58>(v[kk].v[0], E), fx_from_double<58>(v[kk].v[1], E)),
                                     make_longlong2(fx_from_double<58>(v[kk].v[2], E), fx_from_double<58>(v[kk].v[3], E)), a, b);
    });
    *xa = a;
    *xbt = b;
    return E;
}

// The lane's share of delta W (FxW): y_m = D x_m + conj(u_m) G + conj(up) x_{m+1} + dn x_{m-1}
struct FxWLane {
    Limb D, upr, upi, dnr, dni, ur, ui;
    Limb R;
    float Rf;
};

// t <- -i delta W t of NV vectors, one component a lane
template <int NV>
__device__ __forceinline__ void fx_lane_apply(const FxWLane& W, const FxGroup& g, const Limb (&tr)[NV], const Limb (&ti)[NV],
                                              i64 (&outr)[NV], i64 (&outi)[NV]) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const Limb ar = fx_shfl(tr[v], g.up()), ai = fx_shfl(ti[v], g.up());
        const Limb br = fx_shfl(tr[v], g.down()), bi = fx_shfl(ti[v], g.down());
        FxAcc dr = fx_zero<60>(), dn = {0, 0}, di = fx_zero<60>();
        fx_mac(dr, W.ur, tr[v]);
        fx_mac(dn, W.ui, ti[v]);
        fx_mac(di, W.ur, ti[v]);
        fx_mac(di, W.ui, tr[v]);
        const Limb Gr = fx_split(fx_mul_full<55>(W.R, fx_split(g.sum(fx_sum<60>(dr - dn)))));
        const Limb Gi = fx_split(fx_mul_full<55>(W.R, fx_split(g.sum(fx_sum<60>(di)))));
        FxAcc yr = fx_zero<61>(), yi = fx_zero<61>(), nr = {0, 0}, ni = {0, 0};
        fx_mac(yr, W.D, tr[v]);
        fx_mac(yi, W.D, ti[v]);
        fx_mac(yr, W.ur, Gr);
        fx_mac(yr, W.ui, Gi);
        fx_mac(yi, W.ur, Gi);
        fx_mac(ni, W.ui, Gr);
        fx_mac(yr, W.upr, ar);
        fx_mac(yr, W.upi, ai);
        fx_mac(yi, W.upr, ai);
        fx_mac(ni, W.upi, ar);
        fx_mac(yr, W.dnr, br);
        fx_mac(nr, W.dni, bi);
        fx_mac(yi, W.dnr, bi);
        fx_mac(yi, W.dni, br);
        outr[v] = fx_sum<61>(yi - ni);
        outi[v] = -fx_sum<61>(yr - nr);
    }
}

// One fused step of a periodic 1D lattice of L sites held pending K as (P, Q); 30 / LPS sites per warp,
// one warp per CTA.  Numbers and fallback as k_step1d_f64.
template <int VARIANT, int LPS>
__global__ void __launch_bounds__(32) k_step1d_f64_lanes(const double* __restrict__ in, double* __restrict__ out, int L,
                                                         const __grid_constant__ PotConst<double> C, unsigned* status) {
    static_assert(LPS == 5 || LPS == 10, "five or ten lanes per site");
    constexpr int SPW = 30 / LPS, COLS = SPW + 8, NP = 5 * COLS, PER = (NP + 31) / 32, NV = LPS == 5 ? 2 : 1;
    __shared__ longlong2 sp[NP], sq[NP];  // [level][column]
    const int lane = threadIdx.x;
    const int q = lane < 30 ? lane / LPS : SPW - 1;
    const int r = lane < 30 ? lane - LPS * q : lane - 30;
    const int chain = r / 5;  // LPS = 10: 0 psi, 1 d
    const FxGroup g(r % 5, LPS * q + 5 * chain);
    const int x0 = int(blockIdx.x) * SPW;
    const int j = x0 + q < L ? x0 + q : L - 1;
    const bool store = lane < 30 && x0 + q < L;

    double2 v[PER][2];
    unsigned top = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int idx = lane + 32 * i < NP ? lane + 32 * i : NP - 1;
        int x = (x0 - 4 + idx % COLS) % L;
        x = x < 0 ? x + L : x;
        const double2* src = reinterpret_cast<const double2*>(in) + 2 * (int64_t(idx / COLS) * L + x);
        v[i][0] = __ldg(src);
        v[i][1] = __ldg(src + 1);
    }
#pragma unroll
    for (int i = 0; i < PER; ++i)
#pragma unroll
        for (int k = 0; k < 2; ++k) top = max(top, max(fx_hi(v[i][k].x) & 0x7fffffffu, fx_hi(v[i][k].y) & 0x7fffffffu));
    top = __reduce_max_sync(0xffffffffu, top);
    // the FP64 code takes the warp's sites one a lane
    auto in_fp64 = [&]() {
        const int s = x0 + lane;
        const bool own = lane < SPW && s < L;
        const PotConstBase<double> base = C;
        step1d_site_f64<VARIANT, true>(in, out, L, own ? s : j, own, &base, status);
    };
    if (top >= (unsigned(1023 + 50) << 20)) return in_fp64();
    int E = fx_exponent(top);
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (lane + 32 * i < NP) {
            sp[lane + 32 * i] = make_longlong2(fx_from_double<58>(v[i][0].x, E), fx_from_double<58>(v[i][0].y, E));
            sq[lane + 32 * i] = make_longlong2(fx_from_double<58>(v[i][1].x, E), fx_from_double<58>(v[i][1].y, E));
        }
    __syncwarp();
    cpi xa = {0, 0}, xbt = {0, 0};
    static_for<9>([&](auto kc) {
        constexpr int kk = decltype(kc)::value;
        stencil_tap_int<VARIANT, kk>(sp[g.m * COLS + q + kk], sq[g.m * COLS + q + kk], xa, xbt);
    });
    // a site whose K X is more than 2^-7 below the columns' largest (16 times it is 2^62 here) asks for its
    // own exponent
    const int size = g.max_of(max(fx_bits_of(xa.re, xa.im), fx_bits_of(xbt.re, xbt.im)));
    if (top != 0 && __any_sync(0xffffffffu, size < 62 - kFx1dSpread)) E = fx_lane_kinetic_wide<VARIANT>(in, L, j, g, &xa, &xbt);
    xa = {(xa.re + 4) >> 3, (xa.im + 4) >> 3};
    xbt = {(xbt.re + 4) >> 3, (xbt.im + 4) >> 3};
    i64 pr = xa.re + xbt.im, pi = xa.im - xbt.re, dr = xa.re - xbt.im, di = xa.im + xbt.re;

    // U, as fx_unitary with one level a lane
    const int bp = g.max_of(fx_bits_of(pr, pi)), bd0 = g.max_of(fx_bits_of(dr, di));
    const int np = bp ? bp - 58 : -57, nd0 = bd0 ? bd0 - 58 : -57;
    const int nd = nd0 + 1 > np ? nd0 + 1 : np;
    int e = E - 1022 - 55;
    const Limb lpr = fx_split(fx_shift(pr, np)), lpi = fx_split(fx_shift(pi, np));
    FxForms f;
    FxAcc nn = fx_zero<60>();
    fx_mac(nn, lpr, lpr);
    fx_mac(nn, lpi, lpi);
    nn.mid += (fx_mad(lpr.l, lpr.l, 0) >> 32) + (fx_mad(lpi.l, lpi.l, 0) >> 32);
    const i64 n = fx_sum<60>(nn);
    f.rho = g.sum(n);
    f.Fz = g.sum((2 - g.m) * n);
    const Limb r32m1 = fx_split(kFxR32m1);
    {
        const Limb ur = fx_shfl(lpr, g.up()), ui = fx_shfl(lpi, g.up());
        FxAcc a = fx_zero<60>(), b = fx_zero<60>(), n = {0, 0};
        fx_mac(a, lpr, ur);
        fx_mac(a, lpi, ui);
        fx_mac(b, lpr, ui);
        fx_mac(n, lpi, ur);
        i64 fr = fx_sum<60>(a), fi = fx_sum<60>(b - n);
        if (g.m == 1 || g.m == 2) {
            fr += fx_mul(r32m1, fx_split(fr));
            fi += fx_mul(r32m1, fx_split(fi));
        }
        f.Fpr = g.sum(g.m < 4 ? fr : 0);
        f.Fpi = g.sum(g.m < 4 ? fi : 0);
    }
    const int et = e + np - 4;
    const FxBounds bd = fx_bounds(f, et, C.fx);
    if (!__all_sync(0xffffffffu, bd.beta <= kFxBetaMax)) return in_fp64();
    const float beta = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(bd.beta)));
    const int K = fx_degree(beta, kFxTol);
    const int kA = min(K, fx_degree(beta, kFxTolF));
    FxWLane W;
    {
        const i64 gz = fx_coupled(C.fx.dz, f.Fz, et, 0), g2r = fx_coupled(C.fx.dr, f.rho, et, 0);
        W.D = fx_split((2 - g.m) * gz - g2r);
        const i64 er = fx_coupled(C.fx.e0, f.Fpr, et, 1), ei = fx_coupled(C.fx.e0, f.Fpi, et, 1);
        const i64 er1 = er + fx_mul(r32m1, fx_split(er)), ei1 = ei + fx_mul(r32m1, fx_split(ei));
        const bool s_up = g.m == 0 || g.m == 3, s_dn = g.m == 1 || g.m == 4;
        W.upr = fx_split(g.m == 4 ? 0 : (s_up ? er : er1));
        W.upi = fx_split(g.m == 4 ? 0 : (s_up ? ei : ei1));
        W.dnr = fx_split(g.m == 0 ? 0 : (s_dn ? er : er1));
        W.dni = fx_split(g.m == 0 ? 0 : (s_dn ? ei : ei1));
        const Limb mr = fx_shfl(lpr, g.base + 4 - g.m), mi = fx_shfl(lpi, g.base + 4 - g.m);
        auto turned = [&](Limb v) { return (g.m & 1) ? fx_split(-(v.h * (i64(1) << 32) + v.l)) : v; };
        W.ur = turned(mr);
        W.ui = turned(mi);
        fx_singlet(C.fx, et, W.R, W.Rf);
    }
    i64 pc, ps;
    fx_site_phase(f.rho, et, bd.theta, C.fx, pc, ps);
    i64 xr[NV], xi[NV];
    if constexpr (NV == 2) {
        xr[0] = fx_shift(pr, nd);
        xi[0] = fx_shift(pi, nd);
        xr[1] = fx_shift(dr, nd);
        xi[1] = fx_shift(di, nd);
    } else {
        xr[0] = fx_shift(chain ? dr : pr, nd);
        xi[0] = fx_shift(chain ? di : pi, nd);
    }
    Limb tr[NV], ti[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        tr[i] = fx_split(xr[i]);
        ti[i] = fx_split(xi[i]);
    }
#pragma unroll 1
    for (int k = 1; k <= kA; ++k) {
        i64 nr[NV], ni[NV];
        fx_lane_apply<NV>(W, g, tr, ti, nr, ni);
        const Limb fk = fx_inv_fact(k);
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            tr[i] = fx_split(nr[i]);
            ti[i] = fx_split(ni[i]);
            if (k <= 2) {
                xr[i] += k == 1 ? nr[i] : (nr[i] + 1) >> 1;
                xi[i] += k == 1 ? ni[i] : (ni[i] + 1) >> 1;
            } else {
                xr[i] += fx_mul(fk, tr[i]);
                xi[i] += fx_mul(fk, ti[i]);
            }
        }
    }
    if (K > kA) {  // the small terms in FP32
        const float s58 = 3.4694470e-18f, s61 = 4.3368087e-19f;  // 2^-58, 2^-61
        const float fact = s58 * fx_float(fx_inv_fact(kA), s61);
        const float ur = fx_float(W.ur, s58), ui = fx_float(W.ui, s58), D = fx_float(W.D, s61);
        const float upr = fx_float(W.upr, s61), upi = fx_float(W.upi, s61);
        const float dnr = fx_float(W.dnr, s61), dni = fx_float(W.dni, s61);
        FxCpxF t[NV], sum[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            t[i] = {fx_float(tr[i], fact), fx_float(ti[i], fact)};
            sum[i] = {0.f, 0.f};
        }
#pragma unroll 1
        for (int k = kA + 1; k <= K; ++k) {
            const float ik = fx_inv(k);
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const float ar = __shfl_sync(0xffffffffu, t[i].re, g.up()), ai = __shfl_sync(0xffffffffu, t[i].im, g.up());
                const float br = __shfl_sync(0xffffffffu, t[i].re, g.down()), bi = __shfl_sync(0xffffffffu, t[i].im, g.down());
                const float gr = W.Rf * g.sum(fmaf(ur, t[i].re, -ui * t[i].im));
                const float gi = W.Rf * g.sum(fmaf(ur, t[i].im, ui * t[i].re));
                float yr = fmaf(D, t[i].re, fmaf(ur, gr, ui * gi));
                float yi = fmaf(D, t[i].im, fmaf(ur, gi, -ui * gr));
                yr = fmaf(upr, ar, fmaf(upi, ai, yr));
                yi = fmaf(upr, ai, fmaf(-upi, ar, yi));
                yr = fmaf(dnr, br, fmaf(-dni, bi, yr));
                yi = fmaf(dnr, bi, fmaf(dni, br, yi));
                t[i] = {ik * yi, -ik * yr};
                sum[i] = {sum[i].re + t[i].re, sum[i].im + t[i].im};
            }
        }
        const float one = 288230376151711744.f;  // 2^58
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            xr[i] += fx_rint(sum[i].re * one);
            xi[i] += fx_rint(sum[i].im * one);
        }
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        fx_rotate<1>(pc, ps, &xr[i], &xi[i]);
    }
    e += nd - 5;  // 0.5 / 16
    double2* dst = reinterpret_cast<double2*>(out) + 2 * (int64_t(g.m) * L + j);
    if constexpr (NV == 2) {
        const i64 a0 = xr[0] + xr[1], a1 = xi[0] + xi[1], b0 = xr[0] - xr[1], b1 = xi[0] - xi[1];
        if (store) {
            dst[0] = make_double2(fx_pack(a0 - b1, e), fx_pack(a1 + b0, e));
            dst[1] = make_double2(fx_pack(a0 + b1, e), fx_pack(a1 - b0, e));
        }
    } else {  // each half of the lanes stores one of P and Q
        const int other = lane < 30 ? g.base + 5 - 10 * chain + g.m : lane;
        const i64 yr = __shfl_sync(0xffffffffu, xr[0], other), yi = __shfl_sync(0xffffffffu, xi[0], other);
        const i64 psr = chain ? yr : xr[0], psi = chain ? yi : xi[0], dfr = chain ? xr[0] : yr, dfi = chain ? xi[0] : yi;
        const i64 a0 = psr + dfr, a1 = psi + dfi, b0 = psr - dfr, b1 = psi - dfi;
        if (store) dst[chain] = chain ? make_double2(fx_pack(a0 + b1, e), fx_pack(a1 - b0, e))
                                      : make_double2(fx_pack(a0 - b1, e), fx_pack(a1 + b0, e));
    }
}

}  // namespace qlga
