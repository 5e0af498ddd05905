// qlga_step1d_f64.cuh -- the fused 1D FP64 step in integer fixed point.
//
// GB300 issues one FP64 instruction per SM sub-partition every 64-76 cycles (qlga_fixed.cuh); the nine-point
// stencil of K alone is 240 of them a site, 16 k cycles of a warp, longer than all of U on integers.
// K's taps are small integers, so here K runs on integers too, exactly up to the conversion of its
// inputs and one rounding of its sum, and feeds U (fx_unitary) without a conversion in between.
// Of 100 steps with load and read-out, 16384 sites took 4.14 ms in FP64 and 1.48 ms here with five lanes per
// site (below); 1024 sites 1.67 ms, 0.81 ms with ten.
//
// One warp per CTA, one site per lane: small lattices are bound by the latency of one warp's chain,
// so the warps go one to a sub-partition.  A warp loads its 32 columns and the 4-column periodic halo
// on each side (a lane its own column and five values of the halo), converts them and exchanges them
// through shared memory.
//
// Numbers.  Each level has an exponent of its own.  All columns of a level are converted with the largest: components
// below 2^58, so that the stencil's sums (taps of at most 30 in magnitude) fit.  Where K X of a site's level comes
// out more than 2^-6 below that (the edge of a tail, a node), every column takes its own exponent and a lane
// shifts its nine columns to the largest of them.  Either way the rounding is 0.3 of 2^-52 of the largest component
// among the level's nine columns, where FP64 rounds each of the 24 sums at 2^-53.  A warp with a value that
// is not finite, or outside U's domain, takes the FP64 code for both K and U.
#pragma once

#include <cuda_runtime.h>

#include "qlga_batch1d.cuh"
#include "qlga_device.cuh"
#include "qlga_lanes1d.cuh"
#include "qlga_step2d_f64.cuh"  // stencil_tap_int

namespace qlga {

constexpr int kFx1dCols = 40;   // columns a warp reads: 32 and the halo
constexpr int kFx1dSpread = 6;  // a level's K X may lie so many bits below the largest of the warp's columns

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
    __shared__ int se[5][kFx1dCols];
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
    // each level's largest component, of the lane's columns and of the warp's
    unsigned to[5], th[5], tops[5];
    bool fits = true;
    int E[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        to[m] = fx_top(fx_top(fx_top(fx_top(0, own[2 * m].x), own[2 * m].y), own[2 * m + 1].x), own[2 * m + 1].y);
        th[m] = fx_top(0, halo[m]);
        th[m] = max(th[m], __shfl_xor_sync(0xffffffffu, th[m], 1));
        th[m] = max(th[m], __shfl_xor_sync(0xffffffffu, th[m], 2));
        tops[m] = __reduce_max_sync(0xffffffffu, max(to[m], th[m]));
        E[m] = fx_level_exponent(tops[m], fits);
    }
    auto in_fp64 = [&]() {
        const PotConstBase<double> base = C;
        step1d_site_f64<VARIANT, POT>(in, out, L, j, store, &base, status, abi);
    };
    if (!fits) return in_fp64();  // warp-uniform
    auto convert = [&](int m, int Eo, int Eh) {
        sp[m][lane] = make_longlong2(fx_from_double<58>(own[2 * m].x, Eo), fx_from_double<58>(own[2 * m].y, Eo));
        sq[m][lane] = make_longlong2(fx_from_double<58>(own[2 * m + 1].x, Eo), fx_from_double<58>(own[2 * m + 1].y, Eo));
        longlong2* h = hk < 2 ? &sp[m][hc] : &sq[m][hc];
        reinterpret_cast<i64*>(h)[hk & 1] = fx_from_double<58>(halo[m], Eh);
    };
#pragma unroll
    for (int m = 0; m < 5; ++m) convert(m, E[m], E[m]);
    __syncwarp();

    i64 pr[5], pi[5], dr[5], di[5];
    // sum: the lane's (a, bt) of level m, 16 times the true value, in units of 2^(E[m] - 1022 - 58)
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
    bool small = false;  // a level far below the columns' largest (16 times it is 2^62 here)
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        cpi xa = {0, 0}, xbt = {0, 0};
        static_for<9>([&](auto kc) {
            constexpr int kk = decltype(kc)::value;
            stencil_tap_int<VARIANT, kk>(sp[m][lane + kk], sq[m][lane + kk], xa, xbt);
        });
        small = small || (tops[m] != 0 && max(fx_bits_of(xa.re, xa.im), fx_bits_of(xbt.re, xbt.im)) < 62 - kFx1dSpread);
        take(m, xa, xbt);
    }
    if (__any_sync(0xffffffffu, small)) {  // every column with its own exponent, the lane with the largest of its nine
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const int Eo = fx_level_exponent(to[m], fits), Eh = fx_level_exponent(th[m], fits);
            convert(m, Eo, Eh);
            se[m][lane] = Eo;
            if (hk == 0) se[m][hc] = Eh;
        }
        if (!__all_sync(0xffffffffu, fits)) return in_fp64();
        __syncwarp();
        auto down = [](longlong2 v, int n) {
            return make_longlong2((((v.x << 1) >> n) + 1) >> 1, (((v.y << 1) >> n) + 1) >> 1);
        };
#pragma unroll 1
        for (int m = 0; m < 5; ++m) {
            int sh[9], Em = kFxMinExp;
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                sh[k] = se[m][lane + k];
                Em = max(Em, sh[k]);
            }
            cpi xa = {0, 0}, xbt = {0, 0};
            static_for<9>([&](auto kc) {
                constexpr int kk = decltype(kc)::value;
                const int n = min(Em - sh[kk], 63);
                stencil_tap_int<VARIANT, kk>(down(sp[m][lane + kk], n), down(sq[m][lane + kk], n), xa, xbt);
            });
            // m is a run-time value here: the results go through the lane's own row of sp, sq and se
            // once its neighbours have read it
            __syncwarp();
            sp[m][lane] = make_longlong2(xa.re, xa.im);
            sq[m][lane] = make_longlong2(xbt.re, xbt.im);
            se[m][lane] = Em;
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const longlong2 p = sp[m][lane], q = sq[m][lane];
            take(m, cpi{p.x, p.y}, cpi{q.x, q.y});
            E[m] = se[m][lane];
        }
    }

    if (POT) {
        int e[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) e[m] = E[m] - 1022 - 55;
        if (!fx_unitary(pr, pi, dr, di, e, -4, true, C.fx)) return in_fp64();
        if (!store) return;
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const i64 a0 = pr[m] + dr[m], a1 = pi[m] + di[m], b0 = pr[m] - dr[m], b1 = pi[m] - di[m];
            const int eo = e[m] - 5;  // 0.5 / 16
            store_raw_pair(out, int64_t(m) * L + j, fx_pack(a0 - b1, eo), fx_pack(a1 + b0, eo), fx_pack(a0 + b1, eo),
                           fx_pack(a1 - b0, eo));
        }
    } else if (store) {
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const int e = E[m] - 1022 - 58 - 4;
            store_raw_pair(out, int64_t(m) * L + j, fx_pack(pr[m], e), fx_pack(pi[m], e), fx_pack(dr[m], e), fx_pack(di[m], e));
        }
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
    template <class T>
    __device__ __forceinline__ T max_of(T v) const {
        const T s = max(v, __shfl_sync(0xffffffffu, v, s1));
        return max(max(s, __shfl_sync(0xffffffffu, s, s2)), __shfl_sync(0xffffffffu, v, s4));
    }
    __device__ __forceinline__ int up() const { return base + (m < 4 ? m + 1 : 4); }
    __device__ __forceinline__ int down() const { return base + (m > 0 ? m - 1 : 0); }
};

// The lane's level of K at site j with the exponent of its own nine columns (returned; ok: integers can hold them),
// for the warps whose columns have no common one.
template <int VARIANT>
__device__ __noinline__ int fx_lane_kinetic_wide(const double* in, int L, int j, int m, cpi* xa, cpi* xbt, bool* ok) {
    Pair4<double> v[9];
    unsigned top = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        int jj = (j - 4 + k) % L;
        jj = jj < 0 ? jj + L : jj;
        v[k] = load_raw_pair(in, int64_t(m) * L + jj);
#pragma unroll
        for (int q = 0; q < 4; ++q) top = fx_top(top, v[k].v[q]);
    }
    const int E = fx_level_exponent(top, *ok);
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

// The lane's share of delta W (FxW): y_m = D x_m + conj(u_m) G + conj(dn) x_{m+1} + up x_{m-1}, G the sum of v_j x_j
struct FxWLane {
    Limb D, upr, upi, dnr, dni, ur, ui, vr, vi;
};

// t <- -i delta W t of NV vectors, one component a lane
template <int NV>
__device__ __forceinline__ void fx_lane_apply(const FxWLane& W, const FxGroup& g, const Limb (&tr)[NV], const Limb (&ti)[NV],
                                              i64 (&outr)[NV], i64 (&outi)[NV]) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const Limb ar = fx_shfl(tr[v], g.up()), ai = fx_shfl(ti[v], g.up());
        const Limb br = fx_shfl(tr[v], g.down()), bi = fx_shfl(ti[v], g.down());
        FxAcc dr = fx_zero<58>(), dn = {0, 0}, di = fx_zero<58>();
        fx_mac(dr, W.vr, tr[v]);
        fx_mac(dn, W.vi, ti[v]);
        fx_mac(di, W.vr, ti[v]);
        fx_mac(di, W.vi, tr[v]);
        const Limb Gr = fx_split(g.sum(fx_sum<58>(dr - dn))), Gi = fx_split(g.sum(fx_sum<58>(di)));
        FxAcc yr = fx_zero<61>(), yi = fx_zero<61>(), nr = {0, 0}, ni = {0, 0};
        fx_mac(yr, W.D, tr[v]);
        fx_mac(yi, W.D, ti[v]);
        fx_mac(yr, W.ur, Gr);
        fx_mac(yr, W.ui, Gi);
        fx_mac(yi, W.ur, Gi);
        fx_mac(ni, W.ui, Gr);
        fx_mac(yr, W.dnr, ar);
        fx_mac(yr, W.dni, ai);
        fx_mac(yi, W.dnr, ai);
        fx_mac(ni, W.dni, ar);
        fx_mac(yr, W.upr, br);
        fx_mac(nr, W.upi, bi);
        fx_mac(yi, W.upr, bi);
        fx_mac(yi, W.upi, br);
        outr[v] = fx_sum<61>(yi - ni);
        outi[v] = -fx_sum<61>(yr - nr);
    }
}

// fx_log_dot, fx_budget and fx_norm with one level a lane: p, L and T are the lane's level's, pm is p of level -m
__device__ __forceinline__ float fx_lane_log_dot(const FxGroup& g, float pm, float R, float L) {
    const float top = g.max_of(pm + L);
    return R + top + fx_log2(g.sum(fx_exp2(pm + L - top)));
}
__device__ __forceinline__ int fx_lane_budget(const FxGroup& g, float p, float pm, float e_up, float e_dn, float e, float R, float own, float margin) {
    const float ke = fmaxf(0.f, fminf(margin, -kFxLogR32 - e)), ks = fmaxf(0.f, fminf(margin, -R - 2.f * g.max_of(p)));
    float L = own;
#pragma unroll 1
    for (int it = 0; it < 8; ++it) {
        float N = fmaxf(L, fx_lane_log_dot(g, pm, R, L) + ks + pm);
        N = fmaxf(N, e_dn + ke + __shfl_sync(0xffffffffu, L, g.up()));
        N = fmaxf(N, e_up + ke + __shfl_sync(0xffffffffu, L, g.down()));
        if (!__any_sync(0xffffffffu, N > L + 0.01f)) break;
        L = N;
    }
    return int(ceilf(L + 0.001f));
}

// The warp's step in FP64, with the lanes per site that it has: a warp's FP64 instructions cost the same on 3 sites as on
// 32, and one site a lane has ten times as many of them (a field beyond the domain, us a step: 1024
// sites 100, so 34, 16384 sites 431, so 137; the FP64 lane kernel 29 and 171)
template <int VARIANT, int LPS>
__device__ __noinline__ void step1d_lanes_f64(const double* in, double* out, int L, const PotConstBase<double>* C, unsigned* status) {
    lanes1d_step<double, VARIANT, LPS>(in, out, L, *C, status);
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
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int idx = lane + 32 * i < NP ? lane + 32 * i : NP - 1;
        int x = (x0 - 4 + idx % COLS) % L;
        x = x < 0 ? x + L : x;
        const double2* src = reinterpret_cast<const double2*>(in) + 2 * (int64_t(idx / COLS) * L + x);
        v[i][0] = __ldg(src);
        v[i][1] = __ldg(src + 1);
    }
    // each level's largest component among the warp's columns
    unsigned tops[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        unsigned t = 0;
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (lane + 32 * i >= m * COLS && lane + 32 * i < (m + 1) * COLS)
                t = fx_top(fx_top(fx_top(fx_top(t, v[i][0].x), v[i][0].y), v[i][1].x), v[i][1].y);
        tops[m] = __reduce_max_sync(0xffffffffu, t);
    }
    auto in_fp64 = [&]() {
        const PotConstBase<double> base = C;
        step1d_lanes_f64<VARIANT, LPS>(in, out, L, &base, status);
    };
    bool fits = true;
    int Es[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) Es[m] = fx_level_exponent(tops[m], fits);
    if (!fits) return in_fp64();  // warp-uniform
    auto of_level = [](const auto (&a)[5], int m) { return m < 2 ? (m == 0 ? a[0] : a[1]) : (m == 2 ? a[2] : (m == 3 ? a[3] : a[4])); };
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (lane + 32 * i < NP) {
            const int E = of_level(Es, (lane + 32 * i) / COLS);
            sp[lane + 32 * i] = make_longlong2(fx_from_double<58>(v[i][0].x, E), fx_from_double<58>(v[i][0].y, E));
            sq[lane + 32 * i] = make_longlong2(fx_from_double<58>(v[i][1].x, E), fx_from_double<58>(v[i][1].y, E));
        }
    __syncwarp();
    cpi xa = {0, 0}, xbt = {0, 0};
    static_for<9>([&](auto kc) {
        constexpr int kk = decltype(kc)::value;
        stencil_tap_int<VARIANT, kk>(sp[g.m * COLS + q + kk], sq[g.m * COLS + q + kk], xa, xbt);
    });
    int E = of_level(Es, g.m);
    // a level of a site whose K X is more than 2^-kFx1dSpread below the columns' largest (16 times it is 2^62 here)
    // asks for the exponent of its own columns
    const int size = max(fx_bits_of(xa.re, xa.im), fx_bits_of(xbt.re, xbt.im));
    if (__any_sync(0xffffffffu, of_level(tops, g.m) != 0 && size < 62 - kFx1dSpread)) {
        E = fx_lane_kinetic_wide<VARIANT>(in, L, j, g.m, &xa, &xbt, &fits);
        if (!__all_sync(0xffffffffu, fits)) return in_fp64();
    }
    xa = {(xa.re + 4) >> 3, (xa.im + 4) >> 3};
    xbt = {(xbt.re + 4) >> 3, (xbt.im + 4) >> 3};
    i64 pr = xa.re + xbt.im, pi = xa.im - xbt.re, dr = xa.re - xbt.im, di = xa.im + xbt.re;

    // U, as fx_unitary with one level a lane
    const int e = E - 1022 - 55 - 4;  // unit of psi and d
    Limb lpr, lpi;
    int pe;
    fx_level(pr, pi, e, lpr, lpi, pe);
    const float p = fx_log_of(pr, pi, e), own = fmaxf(fmaxf(p, fx_log_of(dr, di, e)), float(kFxFloor));
    const int mirror = g.base + 4 - g.m;
    const int pem = __shfl_sync(0xffffffffu, pe, mirror);
    const float pm = __shfl_sync(0xffffffffu, p, mirror);
    FxForms f;
    f.en = 2 * g.max_of(pe);
    FxAcc nn = fx_zero<60>();
    fx_mac(nn, lpr, lpr);
    fx_mac(nn, lpi, lpi);
    nn.mid += (fx_mad(lpr.l, lpr.l, 0) >> 32) + (fx_mad(lpi.l, lpi.l, 0) >> 32);
    const i64 n = fx_scale_any(fx_sum<60>(nn), 2 * pe - f.en);
    f.rho = g.sum(n);
    f.Fz = g.sum((2 - g.m) * n);
    const Limb r32m1 = fx_split(kFxR32m1);
    {
        const Limb ur = fx_shfl(lpr, g.up()), ui = fx_shfl(lpi, g.up());
        const int pe2 = g.m < 4 ? pe + __shfl_sync(0xffffffffu, pe, g.up()) : (__shfl_sync(0xffffffffu, pe, g.up()), 2 * kFxNone);
        f.fe = g.max_of(pe2);
        FxAcc a = fx_zero<60>(), b = fx_zero<60>(), c = {0, 0};
        fx_mac(a, lpr, ur);
        fx_mac(a, lpi, ui);
        fx_mac(b, lpr, ui);
        fx_mac(c, lpi, ur);
        i64 fr = fx_scale_any(fx_sum<60>(a), pe2 - f.fe), fi = fx_scale_any(fx_sum<60>(b - c), pe2 - f.fe);
        if (g.m == 1 || g.m == 2) {
            fr += fx_mul(r32m1, fx_split(fr));
            fi += fx_mul(r32m1, fx_split(fi));
        }
        f.fr = g.sum(g.m < 4 ? fr : 0);
        f.fi = g.sum(g.m < 4 ? fi : 0);
        fx_coupled_spin(C.fx.e0, f);
    }
    const float le = fx_log_of(f.er, f.ei, f.ee - 60);
    const bool inner_dn = g.m == 1 || g.m == 2, inner_up = g.m == 2 || g.m == 3;  // links with sqrt(3/2)
    const float e_dn = g.m == 4 ? kFxLogNone : (inner_dn ? le + kFxLogR32 : le);
    const float e_up = g.m == 0 ? kFxLogNone : (inner_up ? le + kFxLogR32 : le);
    const float un = fx_pow2f(f.en - 56);
    const float diag = fabsf(fmaf(float(2 - g.m), C.fx.dz_f * un * float(f.Fz), -(C.fx.dr_f * un * float(f.rho))));
    int T = 0;
    float w = 2.f;
#pragma unroll 1
    for (int k = 0; k < kFxMargins; ++k) {
        const int Tk = fx_lane_budget(g, p, pm, e_up, e_dn, le, C.fx.R_log, own, fx_margin(k));
        const float Lt = float(Tk);
        float row = diag + fx_exp2(fx_lane_log_dot(g, pm, C.fx.R_log, Lt) + pm - Lt);
        row += fx_exp2(e_dn + __shfl_sync(0xffffffffu, Lt, g.up()) - Lt);
        row += fx_exp2(e_up + __shfl_sync(0xffffffffu, Lt, g.down()) - Lt);
        const float wk = 1.0001f * g.max_of(row == row ? row : 2.f);
        if (!(w <= kFxNormMax)) {  // all lanes of a site alike
            T = Tk;
            w = wk;
        }
        if (__all_sync(0xffffffffu, w <= kFxNormMax)) break;
    }
    if (!__all_sync(0xffffffffu, w <= kFxNormMax)) return in_fp64();
    const float wmax = fx_warp_max(w);
    FxWLane W;
    {
        const i64 gz = fx_coupled(C.fx.dz, f.Fz, f.en - 56), g2r = fx_coupled(C.fx.dr, f.rho, f.en - 56);
        W.D = fx_split((2 - g.m) * gz - g2r);
        const i64 er1 = f.er + fx_mul(r32m1, fx_split(f.er)), ei1 = f.ei + fx_mul(r32m1, fx_split(f.ei));
        const int su = fx_clamp(f.ee + __shfl_sync(0xffffffffu, T, g.down()) - T + 1, -63, 2);
        const int sd = fx_clamp(f.ee + __shfl_sync(0xffffffffu, T, g.up()) - T + 1, -63, 2);
        W.upr = fx_split(g.m == 0 ? 0 : fx_scale(inner_up ? er1 : f.er, su));
        W.upi = fx_split(g.m == 0 ? 0 : fx_scale(inner_up ? ei1 : f.ei, su));
        W.dnr = fx_split(g.m == 4 ? 0 : fx_scale(inner_dn ? er1 : f.er, sd));
        W.dni = fx_split(g.m == 4 ? 0 : fx_scale(inner_dn ? ei1 : f.ei, sd));
        const Limb mr = fx_shfl(lpr, mirror), mi = fx_shfl(lpi, mirror);
        const int gd = g.max_of(pem + T);
        const int sv = fx_clamp(pem + T - gd, -63, 0), ss = fx_clamp(C.fx.R.ex + pem + gd - T + 3, -63, 5);
        auto turned = [&](i64 x) { return fx_split((g.m & 1) ? -x : x); };
        W.vr = turned(fx_scale(fx_join(mr), sv));
        W.vi = turned(fx_scale(fx_join(mi), sv));
        W.ur = turned(fx_scale(fx_mul_full<60>(C.fx.R.m, mr), ss));
        W.ui = turned(fx_scale(fx_mul_full<60>(C.fx.R.m, mi), ss));
    }
    const int nd = fx_clamp(e + 57 - T, -63, 57);
    i64 pc, ps;
    fx_site_phase(f.rho, f.en - 56, C.fx, pc, ps);
    i64 xr[NV], xi[NV];
    if constexpr (NV == 2) {
        xr[0] = fx_scale(pr, nd);
        xi[0] = fx_scale(pi, nd);
        xr[1] = fx_scale(dr, nd);
        xi[1] = fx_scale(di, nd);
    } else {
        xr[0] = fx_scale(chain ? dr : pr, nd);
        xi[0] = fx_scale(chain ? di : pi, nd);
    }
    Limb tr[NV], ti[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        tr[i] = fx_split(xr[i]);
        ti[i] = fx_split(xi[i]);
    }
    // the terms, as fx_taylor
    auto term_size = [&]() {
        int h = max(fx_abs_limb(tr[0]), fx_abs_limb(ti[0]));
        if constexpr (NV == 2) h = max(h, max(fx_abs_limb(tr[1]), fx_abs_limb(ti[1])));
        return fx_size(fx_warp_max(h));
    };
    float qk = term_size(), fact = 6.9388939e-18f;  // 2^-57
    int k = 0;
#pragma unroll 1
    while (wmax * qk * fx_inv(k + 1) > kFxTolF && k < kFxTerms) {
        ++k;
        fact *= fx_inv(k);
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
        qk = 1.4411519e17f * fact * term_size();  // 2^57
    }
    qk *= wmax * fx_inv(k + 1);
    if (qk > kFxTol) {  // the small terms in FP32
        const float s58 = 3.4694470e-18f, s61 = 4.3368087e-19f;  // 2^-58, 2^-61
        const float ur = fx_float(W.ur, s61), ui = fx_float(W.ui, s61), D = fx_float(W.D, s61);
        const float vr = fx_float(W.vr, s58), vi = fx_float(W.vi, s58);
        const float upr = fx_float(W.upr, s61), upi = fx_float(W.upi, s61);
        const float dnr = fx_float(W.dnr, s61), dni = fx_float(W.dni, s61);
        FxCpxF t[NV], sum[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            t[i] = {fx_float(tr[i], fact), fx_float(ti[i], fact)};
            sum[i] = {0.f, 0.f};
        }
#pragma unroll 1
        while (qk > kFxTol && k < kFxDegree - 1) {
            ++k;
            const float ik = fx_inv(k);
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const float ar = __shfl_sync(0xffffffffu, t[i].re, g.up()), ai = __shfl_sync(0xffffffffu, t[i].im, g.up());
                const float br = __shfl_sync(0xffffffffu, t[i].re, g.down()), bi = __shfl_sync(0xffffffffu, t[i].im, g.down());
                const float gr = g.sum(fmaf(vr, t[i].re, -vi * t[i].im));
                const float gi = g.sum(fmaf(vr, t[i].im, vi * t[i].re));
                float yr = fmaf(D, t[i].re, fmaf(ur, gr, ui * gi));
                float yi = fmaf(D, t[i].im, fmaf(ur, gi, -ui * gr));
                yr = fmaf(dnr, ar, fmaf(dni, ai, yr));
                yi = fmaf(dnr, ai, fmaf(-dni, ar, yi));
                yr = fmaf(upr, br, fmaf(-upi, bi, yr));
                yi = fmaf(upr, bi, fmaf(upi, br, yi));
                t[i] = {ik * yi, -ik * yr};
                sum[i] = {sum[i].re + t[i].re, sum[i].im + t[i].im};
            }
            qk *= wmax * fx_inv(k + 1);
        }
        const float one = 144115188075855872.f;  // 2^57
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
    const int eo = T + 4 - 57 - 5;  // 0.5 / 16 of the unnormalised result
    double2* dst = reinterpret_cast<double2*>(out) + 2 * (int64_t(g.m) * L + j);
    if constexpr (NV == 2) {
        const i64 a0 = xr[0] + xr[1], a1 = xi[0] + xi[1], b0 = xr[0] - xr[1], b1 = xi[0] - xi[1];
        if (store) {
            dst[0] = make_double2(fx_pack(a0 - b1, eo), fx_pack(a1 + b0, eo));
            dst[1] = make_double2(fx_pack(a0 + b1, eo), fx_pack(a1 - b0, eo));
        }
    } else {  // each half of the lanes stores one of P and Q
        const int other = lane < 30 ? g.base + 5 - 10 * chain + g.m : lane;
        const i64 yr = __shfl_sync(0xffffffffu, xr[0], other), yi = __shfl_sync(0xffffffffu, xi[0], other);
        const i64 psr = chain ? yr : xr[0], psi = chain ? yi : xi[0], dfr = chain ? xr[0] : yr, dfi = chain ? xi[0] : yi;
        const i64 a0 = psr + dfr, a1 = psi + dfi, b0 = psr - dfr, b1 = psi - dfi;
        if (store) dst[chain] = chain ? make_double2(fx_pack(a0 + b1, eo), fx_pack(a1 - b0, eo))
                                      : make_double2(fx_pack(a0 - b1, eo), fx_pack(a1 + b0, eo));
    }
}

}  // namespace qlga
