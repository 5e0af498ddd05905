// qlga_adjoint2d_f64.cuh -- K^dagger of a 2D FP64 lattice in integer fixed point, both axes in one pass.
//
// The adjoint of k_kinetic2d_f64 (qlga_step2d_f64.cuh): warp strips of one level that march along y.  K = K_y K_x, so
// y comes first here: each lane runs the four adjoint blocks of y as a register pipeline on its column, lanes 0
// to 7 also on the eight columns beyond, the row goes to shared memory, and the adjoint nine-point stencil
// of x reads it there.  The FP64 form was two passes of 320 FP64 instructions a site (66 cycles each): 106 us at 256^2, 29 here, and 78
// where the cores of a vortex lattice send strips to FP64.
//
// Numbers.  As there, with components below 2^57 after conversion: the y blocks' taps (at most 44 in magnitude) keep
// below 2^63, are rounded to 2^-5 of that, and the x stencil's sums, below 2^63 again, are eight times the true K^dagger g.
// The rounding is 2^-57.1 (root mean square) of a strip's largest, so the same spread of a strip's columns sends its
// chunk to FP64: the cotangent of a local loss keeps its tails.
#pragma once

#include "qlga_adjoint.cuh"
#include "qlga_step2d_f64.cuh"

namespace qlga {

// One adjoint block C^dagger S_c C'^dagger S_c^T along y for one component (make_stencil_adjoint has the same
// factors): input row n -> output row n - 1; yo: the other qubit of the previous row, wc: the shifted qubit after the
// first collide of the previous row.
template <int C, int FIRST, class N>
__device__ __forceinline__ void stream_adj(N& a, N& bt, N& yo, N& wc) {
    const N ya = C == 1 ? yo : a, yb = C == 1 ? bt : yo;
    yo = C == 1 ? a : bt;
    const N wa = ya - yb, wb = ya + yb;
    const N za = C == 1 ? wa : wc, zb = C == 1 ? wc : wb;
    wc = C == 1 ? wb : wa;
    a = FIRST == 0 ? za - zb : za + zb;
    bt = FIRST == 0 ? za + zb : zb - za;
}

template <class P>
struct AdjColumn {  // P: a pair of numbers, re and im
    P yo[4], wc[4];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int k = 0; k < 4; ++k) yo[k] = wc[k] = {0, 0};
    }
    template <int VARIANT>
    __device__ __forceinline__ void push(P& a, P& bt) {
        static_for<4>([&](auto kc) {
            constexpr int kk = decltype(kc)::value, c = kk < 2 ? 0 : 1;  // the blocks of qubit 1 first
            stream_adj<c, VARIANT>(a.re, bt.re, yo[kk].re, wc[kk].re);
            stream_adj<c, VARIANT>(a.im, bt.im, yo[kk].im, wc[kk].im);
        });
    }
};
struct AdjColumnInt : AdjColumn<cpi> {
    __device__ __forceinline__ void scale(int n) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            yo[k] = {strip_scale(yo[k].re, n), strip_scale(yo[k].im, n)};
            wc[k] = {strip_scale(wc[k].re, n), strip_scale(wc[k].im, n)};
        }
    }
    template <int VARIANT>
    __device__ __forceinline__ void push_rounded(longlong2& a, longlong2& bt) {
        cpi x = {a.x, a.y}, y = {bt.x, bt.y};
        push<VARIANT>(x, y);
        auto down = [](i64 v) { return ((v >> 4) + 1) >> 1; };
        a = make_longlong2(down(x.re), down(x.im));
        bt = make_longlong2(down(y.re), down(y.im));
    }
};

// The chunk of one warp in FP64: rows [y_begin, y_end) of its 32 columns of one level, straight from global memory;
// yrow: the warp's row in shared memory.
template <int VARIANT>
__device__ __noinline__ void adjoint_strip_f64(const double2* level, double2* out2, int nx, int ny, int x0, int y_begin,
                                               int y_end, double2* yrow) {
    constexpr KinStencil S = kStencilAdj[VARIANT];
    const int lane = threadIdx.x & 31;
    auto wrap = [&](int x) { return (x % nx + nx) % nx; };
    const int xm = wrap(x0 - kStep2dHalo + lane), xh = wrap(x0 + kStep2dWarpCols - kStep2dHalo + (lane & 7));
    AdjColumn<cpx<double>> own, beyond;
    own.clear();
    beyond.clear();
    const int nrows = (y_end - y_begin) + 8;
#pragma unroll 1
    for (int r = 0; r < nrows; ++r) {
        int y = y_begin - kStep2dHalo + r;
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        const double2* g = level + 2 * int64_t(y) * nx;
        auto column = [&](AdjColumn<cpx<double>>& c, int x, int at) {
            const double2 u = __ldg(g + 2 * x), v = __ldg(g + 2 * x + 1);
            cpx<double> a = {u.x, u.y}, bt = {v.x, v.y};
            c.template push<VARIANT>(a, bt);
            yrow[2 * at] = make_double2(a.re, a.im);
            yrow[2 * at + 1] = make_double2(bt.re, bt.im);
        };
        __syncwarp();  // the last row's stencil has read yrow
        column(own, xm, lane);
        if (lane < 2 * kStep2dHalo) column(beyond, xh, kStep2dWarpCols + lane);
        __syncwarp();
        if (r < 8) continue;
        cpx<double> xa = {0.0, 0.0}, xbt = {0.0, 0.0};
        static_for<9>([&](auto kc) {
            constexpr int kk = decltype(kc)::value;
            const double2 P = yrow[2 * (lane + kk)], Q = yrow[2 * (lane + kk) + 1];
            kin_tap4<S.g[0][0][kk], S.g[0][1][kk], S.g[1][0][kk], S.g[1][1][kk]>(cpx<double>{P.x, P.y}, cpx<double>{Q.x, Q.y}, xa, xbt);
        });
        if (x0 + lane < nx) {
            const double s = 1.0 / 256.0;
            double2* p2 = out2 + 2 * (int64_t(y_begin + r - 8) * nx + x0 + lane);
            p2[0] = make_double2(s * xa.re, s * xa.im);
            p2[1] = make_double2(s * xbt.re, s * xbt.im);
        }
    }
}

constexpr int kAdj64Ctas = 4;  // resident per SM, of kKin64Warps warps

// out = K^dagger in, both in the resident layout (a, bt); strips, chunks and their FP64 form as in
// k_kinetic2d_f64.
template <int VARIANT>
__global__ void __launch_bounds__(32 * kKin64Warps, kAdj64Ctas)
    k_adjoint2d_f64(const double* __restrict__ in, double* __restrict__ out, int nx, int ny, int chunks) {
    constexpr KinStencil S = kStencilAdj[VARIANT];
    constexpr int kRow = kStep2dWarpRowSites * 2;  // double2 of a row
    __shared__ double2 ring_all[kKin64Warps][kKin64Stages][kRow];
    __shared__ longlong2 yrow_all[kKin64Warps][kRow];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int strips = (nx + kStep2dWarpCols - 1) / kStep2dWarpCols;
    const int64_t gw = int64_t(blockIdx.x) * kKin64Warps + w;
    if (gw >= 5 * int64_t(strips) * chunks) return;  // whole warp: no block-wide barrier follows
    const int m = int(gw % 5);
    const int strip = int(gw / 5) % strips, chunk = int(gw / 5) / strips;
    const int x0 = strip * kStep2dWarpCols;
    const int y_begin = int((int64_t(chunk) * ny) / chunks);
    const int y_end = int((int64_t(chunk + 1) * ny) / chunks);
    const int64_t nsites = int64_t(nx) * ny;
    const double2* level = reinterpret_cast<const double2*>(in) + 2 * (m * nsites);
    double2* out2 = reinterpret_cast<double2*>(out) + 2 * (m * nsites);
    double2(*ring)[kRow] = ring_all[w];
    longlong2* yrow = yrow_all[w];

    const int nrows = (y_end - y_begin) + 8;
    auto wrap_x = [&](int x) {  // x < nx + 36 < 3 nx
        x = x < 0 ? x + nx : x;
        x = x >= nx ? x - nx : x;
        return x >= nx ? x - nx : x;
    };
    const int xm = wrap_x(x0 - kStep2dHalo + lane);
    const int xh = wrap_x(x0 + kStep2dWarpCols - kStep2dHalo + lane);
    int y_in = y_begin - kStep2dHalo, issued = 0;
    y_in = y_in < 0 ? y_in + ny : y_in;
    auto issue_row = [&]() {  // the next row, if there is one
        if (issued < nrows) {
            double2* d = ring[issued % kKin64Stages] + 2 * lane;
            const double2* g = level + 2 * (int64_t(y_in) * nx + xm);
            cp_async_16(d, g);
            cp_async_16(d + 1, g + 1);
            if (lane < 2 * kStep2dHalo) {
                const double2* h = level + 2 * (int64_t(y_in) * nx + xh);
                cp_async_16(d + 2 * kStep2dWarpCols, h);
                cp_async_16(d + 2 * kStep2dWarpCols + 1, h + 1);
            }
            y_in = y_in + 1 == ny ? 0 : y_in + 1;
            ++issued;
        }
        cp_async_commit();
    };
#pragma unroll
    for (int r = 0; r < kKin64Stages - 1; ++r) issue_row();

    AdjColumnInt own, beyond;
    own.clear();
    beyond.clear();
    int E = kFxMinExp;                              // the pipelines' exponent
    int seen = kFxMinExp, seen_before = kFxMinExp;  // the largest row exponents of this and the last 8 rows
    int low = 2047, low_before = 2047;              // and the smallest exponents of four neighbours

#pragma unroll 1
    for (int r = 0; r < nrows; ++r) {
        cp_async_wait<kKin64Stages - 2>();
        __syncwarp();
        issue_row();

        double2* row = ring[r % kKin64Stages];
        const double2 own0 = row[2 * lane], own1 = row[2 * lane + 1];
        double2* tail = row + 2 * kStep2dWarpCols;  // columns 32..39: the lane's component
        const double halo = reinterpret_cast<const double*>(tail)[lane];
        auto hi = [](double x) { return fx_hi(x) & 0x7fffffffu; };
        const unsigned column = max(max(hi(own0.x), hi(own0.y)), max(hi(own1.x), hi(own1.y)));
        const unsigned top = __reduce_max_sync(0xffffffffu, max(column, hi(halo)));
        const int Er = fx_exponent(top);
        if ((r & 7) == 0) {
            seen_before = seen;
            seen = kFxMinExp;
            low_before = low;
            low = 2047;
        }
        seen = max(seen, Er);
        if (top) low = min(low, strip_low(column, hi(halo)));  // an empty row adds nothing to any site
        const int En = max(seen, seen_before);
        if (En - min(low, low_before) > kKin64Spread || En > kKin64MaxExp) {  // warp-uniform
            cp_async_wait<0>();
            adjoint_strip_f64<VARIANT>(level, out2, nx, ny, x0, y_begin, y_end, reinterpret_cast<double2*>(yrow));
            return;
        }
        if (En != E) {  // warp-uniform, rare on smooth fields
            const int n = max(E - En, -63);
            own.scale(n);
            beyond.scale(n);
            E = En;
        }
        longlong2 a = make_longlong2(fx_from_double<57>(own0.x, E), fx_from_double<57>(own0.y, E));
        longlong2 bt = make_longlong2(fx_from_double<57>(own1.x, E), fx_from_double<57>(own1.y, E));
        reinterpret_cast<i64*>(tail)[lane] = fx_from_double<57>(halo, E);
        __syncwarp();  // also: the last row's stencil has read yrow
        own.push_rounded<VARIANT>(a, bt);
        yrow[2 * lane] = a;
        yrow[2 * lane + 1] = bt;
        if (lane < 2 * kStep2dHalo) {
            const longlong2* h = reinterpret_cast<const longlong2*>(tail) + 2 * lane;
            longlong2 ha = h[0], hb = h[1];
            beyond.push_rounded<VARIANT>(ha, hb);
            yrow[2 * (kStep2dWarpCols + lane)] = ha;
            yrow[2 * (kStep2dWarpCols + lane) + 1] = hb;
        }
        if (r < 8) continue;  // the pipelines fill
        __syncwarp();
        cpi xa = {0, 0}, xbt = {0, 0};
        const longlong2* p = yrow + 2 * lane;
        static_for<9>([&](auto kc) {
            constexpr int kk = decltype(kc)::value;
            const longlong2 P = p[2 * kk], Q = p[2 * kk + 1];
            xa.re = tap_int<S.g[0][1][kk]>(Q.x, tap_int<S.g[0][0][kk]>(P.x, xa.re));
            xa.im = tap_int<S.g[0][1][kk]>(Q.y, tap_int<S.g[0][0][kk]>(P.y, xa.im));
            xbt.re = tap_int<S.g[1][1][kk]>(Q.x, tap_int<S.g[1][0][kk]>(P.x, xbt.re));
            xbt.im = tap_int<S.g[1][1][kk]>(Q.y, tap_int<S.g[1][0][kk]>(P.y, xbt.im));
        });
        if (x0 + lane < nx) {  // output row y_begin + r - 8
            double2* p2 = out2 + 2 * (int64_t(y_begin + r - 8) * nx + x0 + lane);
            const FxToDouble to(E - 1022 - 60);
            p2[0] = make_double2(to(xa.re), to(xa.im));
            p2[1] = make_double2(to(xbt.re), to(xbt.im));
        }
    }
    cp_async_wait<0>();
}

}  // namespace qlga
