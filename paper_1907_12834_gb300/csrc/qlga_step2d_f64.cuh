// qlga_step2d_f64.cuh -- the 2D FP64 kinetic operator in integer fixed point.
//
// K along x and y in one pass, by the y-marching warp strips of qlga_step2d.cuh, a level to a warp: a warp owns
// 32 columns of one level and a row range, stages rows (with the 4-column periodic halo) in its own cp.async ring,
// applies the nine-point x stencil from shared memory and runs the four y blocks as a register pipeline.  All
// of K's coefficients are small integers, so on integers K is exact up to one rounding between the
// axes, and an addition costs 2 cycles per sub-partition where FP64 takes 76 (qlga_fixed.cuh): at 1024^2 the
// pass takes 0.14 ms (K in FP64 1.36; all levels of a strip in one warp, with 255 registers and 8 warps per SM, 0.187),
// 20 us at 256^2.
// The potential is a pass of its own (k_potential): FP64 state traffic is far
// from the bound.
//
// Numbers.  A row is converted once, in place in the ring, each lane its column and an equal share of
// the eight halo columns, to int64 with one exponent per warp: components below 2^58, the largest of
// the last 8 to 16 rows in [2^57, 2^58) when its row was read.  The stencil's taps sum to at most 30
// in magnitude, so its sums fit; they are rounded to 2^-6 of their unit, and the y blocks (taps at
// most 44) then end below 2^63 and hold four times the true K X.  Where a row is larger than all before it the
// pipeline is shifted down, where the last 16 rows are smaller it is shifted up.  The rounding is
// thus 2^-57.2 (root mean square) of the largest component of the level in a strip of 40 columns and 8 to 16 rows, where
// FP64 adds 2^-53 of what lies within the stencil.  A warp whose strip varies by more than the difference redoes
// its chunk in FP64: one that meets four neighbouring columns more than 2^-kKin64Spread below the largest
// (the tail of a localised state), where any nine columns hold four such neighbours.
#pragma once

#include <cuda_runtime.h>

#include "qlga_device.cuh"
#include "qlga_step2d.cuh"  // cp.async helpers, strip geometry

namespace qlga {

// acc + c x for a compile-time integer c, by shifts and additions
template <int C>
__device__ __forceinline__ i64 tap_int(i64 x, i64 acc) {
    if constexpr (C == 0) return acc;
    else if constexpr (C < 0) {
        if constexpr (C == -1) return acc - x;
        else if constexpr (C == -3) return acc - x - (x << 1);
        else if constexpr (C == -5) return acc - x - (x << 2);
        else return acc - i64(-C) * x;
    } else {
        if constexpr (C == 1) return acc + x;
        else if constexpr (C == 3) return acc + x + (x << 1);
        else if constexpr (C == 5) return acc + x + (x << 2);
        else return acc + i64(C) * x;
    }
}

struct cpi {
    i64 re, im;
};

// One tap of the x stencil on a staged (P, Q) pair (re and im of each).
template <int VARIANT, int K>
__device__ __forceinline__ void stencil_tap_int(const longlong2 P, const longlong2 Q, cpi& xa, cpi& xbt) {
    constexpr KinStencil S = kStencilPQ[VARIANT];
    xa.re = tap_int<S.g[0][1][K]>(Q.x, tap_int<S.g[0][0][K]>(P.x, xa.re));
    xa.im = tap_int<S.g[0][1][K]>(Q.y, tap_int<S.g[0][0][K]>(P.y, xa.im));
    xbt.re = tap_int<S.g[1][1][K]>(Q.x, tap_int<S.g[1][0][K]>(P.x, xbt.re));
    xbt.im = tap_int<S.g[1][1][K]>(Q.y, tap_int<S.g[1][0][K]>(P.y, xbt.im));
}

// One streaming block along y for one component of one level (stream_block, qlga_step2d.cuh).
template <int C, int FIRST>
__device__ __forceinline__ void stream_int(i64& a, i64& bt, i64& yo, i64& wc) {
    const i64 ia = a, ibt = bt;
    if (C == 1) {
        const i64 ybt = FIRST == 0 ? ibt - ia : ia + ibt;
        const i64 wa = yo + ybt, wbt = ybt - yo;
        yo = FIRST == 0 ? ia + ibt : ia - ibt;
        a = wa;
        bt = wc;
        wc = wbt;
    } else {
        const i64 ya = FIRST == 0 ? ia + ibt : ia - ibt;
        const i64 wa = ya + yo, wbt = yo - ya;
        yo = FIRST == 0 ? ibt - ia : ia + ibt;
        a = wc;
        bt = wbt;
        wc = wa;
    }
}

constexpr int kKin64Warps = 4;  // of a CTA: one to a sub-partition
constexpr int kKin64Ctas = 5;   // resident per SM
constexpr int kKin64Stages = 3;
constexpr int kKin64Spread = 4;
// The smallest exponent of four neighbouring columns of a row (aligned with the strip), from the largest high words
// of the lane's own column and of its halo component; 0 where such four are empty.  All lanes take part.
__device__ __forceinline__ int strip_low(unsigned column, unsigned halo) {
    column = max(column, __shfl_xor_sync(0xffffffffu, column, 1));
    column = max(column, __shfl_xor_sync(0xffffffffu, column, 2));
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) halo = max(halo, __shfl_xor_sync(0xffffffffu, halo, o));  // four lanes hold a column
    return int(__reduce_min_sync(0xffffffffu, min(column, halo)) >> 20);
}
// v 2^n, rounded, for the pipelines' values (up to 2^63)
QLGA_HD i64 strip_scale(i64 v, int n) { return n > 0 ? v << n : (n < 0 ? ((v >> (-n - 1)) + 1) >> 1 : v); }

constexpr int kKin64MaxExp = 1022 + 900;  // larger components, and those that are not finite, take FP64

// The chunk of one warp in FP64: rows [y_begin, y_end) of its 32 columns of one level, straight from global memory.
template <int VARIANT>
__device__ __noinline__ void kinetic_strip_f64(const double2* level, double2* out2, int nx, int ny, int x0, int y_begin,
                                               int y_end, bool abi) {
    const int lane = threadIdx.x & 31;
    const int xc = (x0 + lane) % nx;
    cpx<double> yo[4], wc[4];
    for (int k = 0; k < 4; ++k) yo[k] = wc[k] = {0.0, 0.0};
    const int nrows = (y_end - y_begin) + 8;
#pragma unroll 1
    for (int r = 0; r < nrows; ++r) {
        int y = y_begin - kStep2dHalo + r;
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        cpx<double> xa = {0.0, 0.0}, xbt = {0.0, 0.0};
        static_for<9>([&](auto kc) {
            constexpr int kk = decltype(kc)::value;
            constexpr KinStencil S = kStencilPQ[VARIANT];
            int x = xc + kk - 4;
            x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
            const double2* g = level + 2 * (int64_t(y) * nx + x);
            const double2 P = __ldg(g), Q = __ldg(g + 1);
            kin_tap4<S.g[0][0][kk], S.g[0][1][kk], S.g[1][0][kk], S.g[1][1][kk]>(cpx<double>{P.x, P.y}, cpx<double>{Q.x, Q.y}, xa, xbt);
        });
        static_for<4>([&](auto kc) {  // stream_block, qlga_step2d.cuh
            constexpr int kk = decltype(kc)::value;
            const cpx<double> ia = xa, ibt = xbt;
            if (kk < 2) {
                const cpx<double> ybt = VARIANT == 0 ? ibt - ia : ia + ibt;
                const cpx<double> wa = yo[kk] + ybt, wbt = ybt - yo[kk];
                yo[kk] = VARIANT == 0 ? ia + ibt : ia - ibt;
                xa = wa;
                xbt = wc[kk];
                wc[kk] = wbt;
            } else {
                const cpx<double> ya = VARIANT == 0 ? ia + ibt : ia - ibt;
                const cpx<double> wa = ya + yo[kk], wbt = yo[kk] - ya;
                yo[kk] = VARIANT == 0 ? ibt - ia : ia + ibt;
                xa = wc[kk];
                xbt = wbt;
                wc[kk] = wa;
            }
        });
        if (r >= 8 && x0 + lane < nx) {
            const double s = 1.0 / 256.0;
            double2* p2 = out2 + 2 * (int64_t(y_begin + r - 8) * nx + x0 + lane);
            p2[0] = make_double2(s * xa.re, s * xa.im);
            p2[1] = abi ? make_double2(s * xbt.im, -(s * xbt.re)) : make_double2(s * xbt.re, s * xbt.im);
        }
    }
}

// out = K in: in held pending K as (P, Q), out the true state in the resident layout (a, bt) or,
// with abi, the ABI's (a, b).  nx >= 32
// of any remainder: the lanes of the last strip that lie past the row's end work on its periodic
// image and store nothing.
template <int VARIANT>
__global__ void __launch_bounds__(32 * kKin64Warps, kKin64Ctas)
    k_kinetic2d_f64(const double* __restrict__ in, double* __restrict__ out, int nx, int ny, int chunks, bool abi) {
    constexpr int kRow = kStep2dWarpRowSites * 2;  // double2 of a row
    __shared__ double2 ring_all[kKin64Warps][kKin64Stages][kRow];
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

    cpi yo[4], wc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) yo[k] = wc[k] = {0, 0};
    int E = kFxMinExp;                              // the pipeline's exponent
    int seen = kFxMinExp, seen_before = kFxMinExp;  // the largest row exponents of this and the last 8 rows
    int low = 2047, low_before = 2047;              // and the smallest exponents of four neighbours

#pragma unroll 1
    for (int r = 0; r < nrows; ++r) {
        cp_async_wait<kKin64Stages - 2>();
        __syncwarp();
        issue_row();

        double2* row = ring[r % kKin64Stages];
        // convert the row in place: column `lane` of the ring and the lane's component of columns 32..39
        const double2 own0 = row[2 * lane], own1 = row[2 * lane + 1];
        const double halo = reinterpret_cast<const double*>(row + 2 * kStep2dWarpCols)[lane];
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
            kinetic_strip_f64<VARIANT>(level, out2, nx, ny, x0, y_begin, y_end, abi);
            return;
        }
        if (En != E) {  // warp-uniform, rare on smooth fields
            const int n = max(E - En, -63);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                yo[k] = {strip_scale(yo[k].re, n), strip_scale(yo[k].im, n)};
                wc[k] = {strip_scale(wc[k].re, n), strip_scale(wc[k].im, n)};
            }
            E = En;
        }
        longlong2* p = reinterpret_cast<longlong2*>(row + 2 * lane);
        p[0] = make_longlong2(fx_from_double<58>(own0.x, E), fx_from_double<58>(own0.y, E));
        p[1] = make_longlong2(fx_from_double<58>(own1.x, E), fx_from_double<58>(own1.y, E));
        reinterpret_cast<i64*>(row + 2 * kStep2dWarpCols)[lane] = fx_from_double<58>(halo, E);
        __syncwarp();

        // x axis: nine-point stencil (x16) from the held (P, Q) pairs to (a, bt), then rounded to 2^-6
        cpi xa = {32, 32}, xbt = {32, 32};
        static_for<9>([&](auto kc) {
            constexpr int kk = decltype(kc)::value;
            stencil_tap_int<VARIANT, kk>(p[2 * kk], p[2 * kk + 1], xa, xbt);
        });
        xa = {xa.re >> 6, xa.im >> 6};
        xbt = {xbt.re >> 6, xbt.im >> 6};
        // y axis: I'_2 I'_2 then I'_1 I'_1 as a streaming pipeline (x16: four times the true K X)
        static_for<4>([&](auto kc) {
            constexpr int kk = decltype(kc)::value;
            stream_int<kk < 2 ? 1 : 0, VARIANT>(xa.re, xbt.re, yo[kk].re, wc[kk].re);
            stream_int<kk < 2 ? 1 : 0, VARIANT>(xa.im, xbt.im, yo[kk].im, wc[kk].im);
        });
        if (r >= 8 && x0 + lane < nx) {  // pipeline full: this is output row y_begin + r - 8
            double2* p2 = out2 + 2 * (int64_t(y_begin + r - 8) * nx + x0 + lane);
            const FxToDouble to(E - 1022 - 60);
            p2[0] = make_double2(to(xa.re), to(xa.im));
            p2[1] = abi ? make_double2(to(xbt.im), to(-xbt.re)) : make_double2(to(xbt.re), to(xbt.im));
        }
    }
    cp_async_wait<0>();
}

}  // namespace qlga
