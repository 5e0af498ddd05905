// qlga_adjoint_kernel.cuh -- the kernel of one axis of K^dagger with the pull-back through U (qlga_adjoint.cuh, and in
// integer fixed point for an FP64 state, qlga_fixed_adjoint.cuh).
#pragma once

#include "qlga_adjoint.cuh"
#include "qlga_fixed_adjoint.cuh"

namespace qlga {

constexpr int kAdjThreads = 128;

// Per-thread sum of the per-site coupling-gradient terms: FP64 for an FP64 state; compensated
// (Kahan) FP32 for an FP32 state, whose terms carry FP32 rounding anyway and whose FP64 additions
// would cost 64 FP32 slots each.  Block sums are FP64.
template <class T>
struct AdjSum;
template <>
struct AdjSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double v) { s += v; }
    __device__ __forceinline__ double value() const { return s; }
};
template <>
struct AdjSum<float> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float y = v - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return double(s) - double(c); }
};

// Resident pair (a, bt) of level m at a site.
template <class T>
__device__ __forceinline__ void load_resident(const T* X, int64_t nsites, int m, int64_t site, cpx<T>& a,
                                              cpx<T>& bt) {
    if constexpr (sizeof(T) == 4) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(X) + m * nsites + site);
        a = {v.x, v.y};
        bt = {v.z, v.w};
    } else {
        const double2* p = reinterpret_cast<const double2*>(X) + 2 * (m * nsites + site);
        const double2 u = __ldg(p), w = __ldg(p + 1);
        a = {u.x, u.y};
        bt = {w.x, w.y};
    }
}

// The FP64 pull-back for the warps that the fixed-point form leaves: a call, so that the kernel keeps its registers.
__device__ __noinline__ void potential_vjp_f64(const cpx<double>* a, const cpx<double>* b, cpx<double>* ga, cpx<double>* gb,
                                               const AdjConst<double>* A, double* dc, unsigned* status) {
    potential_vjp_site<double>(a, b, ga, gb, *A, dc, status);
}

// gout = [U_X^T o] K_axis^dagger gin on resident cotangent buffers: the adjoint nine-point
// stencil of one axis, optionally followed by the pull-back through U at the state X (resident,
// the true state before U).  VJP: dL/dg of this launch is added to partials[block][3] (each block
// owns its row, so repeated launches with the same grid accumulate deterministically).
// LOCAL (with VJP): gin is K^dagger g already (k_adjoint2d_f64), and only the pull-back through U follows.
template <class T, int VARIANT, bool VJP, bool LOCAL = false>
// FP32: 4 resident CTAs per SM (128 registers, a few spilled) beat 3 at 168 registers by 12%.
__global__ void __launch_bounds__(kAdjThreads, sizeof(T) == 4 ? 4 : 1) k_adjoint_axis(const T* __restrict__ gin, T* __restrict__ gout,
                                                              const T* __restrict__ X, int64_t nx, int64_t ny,
                                                              int axis, AdjConst<T> A,
                                                              double* __restrict__ partials, unsigned* status) {
    constexpr KinStencil S = kStencilAdj[VARIANT];
    const int64_t nsites = nx * ny;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    AdjSum<T> dsum[3];
    for (int64_t base = int64_t(blockIdx.x) * blockDim.x; base < nsites; base += stride) {
        const int64_t site = base + threadIdx.x;
        const bool active = site < nsites;
        const int64_t s = active ? site : 0;
        const int64_t x = s % nx, y = s / nx;
        int64_t nb[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            if (axis == 0) {
                int64_t xx = x + k - 4;
                xx = xx < 0 ? xx + nx : (xx >= nx ? xx - nx : xx);
                nb[k] = y * nx + xx;
            } else {
                int64_t yy = y + k - 4;
                yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
                nb[k] = yy * nx + x;
            }
        }
        cpx<T> ga[5], gb[5];
        if (LOCAL) SiteIO<T>::load(gin, nsites, s, ga, gb);
#pragma unroll
        for (int m = 0; m < (LOCAL ? 0 : 5); ++m) {
            cpx<T> acc_a = {T(0), T(0)}, acc_bt = {T(0), T(0)};
            static_for<9>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                cpx<T> a, bt;
                load_resident(gin, nsites, m, nb[k], a, bt);
                kin_tap4<S.g[0][0][k], S.g[0][1][k], S.g[1][0][k], S.g[1][1][k]>(a, bt, acc_a, acc_bt);
            });
            const T sc = T(0.0625);
            ga[m] = {sc * acc_a.re, sc * acc_a.im};
            gb[m] = {sc * acc_bt.im, -sc * acc_bt.re};  // b = -i bt
        }
        if (VJP) {
            cpx<T> a[5], b[5];
            SiteIO<T>::load(X, nsites, s, a, b);
            T dc[3];
            if constexpr (std::is_same<T, double>::value) {
                // the CTA's warps run the long site code together, for the instruction cache (a gradient of
                // 512^2 25.2 ms, 27.7 without)
                __syncthreads();
                if (!fx_vjp_site(a, b, ga, gb, A, dc)) {  // warp-uniform
                    cpx<double> v[4][5];
#pragma unroll
                    for (int m = 0; m < 5; ++m) {
                        v[0][m] = a[m];
                        v[1][m] = b[m];
                        v[2][m] = ga[m];
                        v[3][m] = gb[m];
                    }
                    const AdjConst<double> Ac = A;
                    potential_vjp_f64(v[0], v[1], v[2], v[3], &Ac, dc, status);
#pragma unroll
                    for (int m = 0; m < 5; ++m) {
                        ga[m] = v[2][m];
                        gb[m] = v[3][m];
                    }
                }
            } else {
                potential_vjp_site(a, b, ga, gb, A, dc, status);
            }
            if (active) {
                dsum[0].add(dc[0]);
                dsum[1].add(dc[1]);
                dsum[2].add(dc[2]);
            }
        }
        if (active) SiteIO<T>::store(gout, nsites, site, ga, gb);
    }
    if (VJP) {
        __shared__ double sh[kAdjThreads / 32][3];
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            double v = dsum[j].value();
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) sh[wid][j] = v;
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            double v = 0.0;
            for (int w = 0; w < kAdjThreads / 32; ++w) v += sh[w][threadIdx.x];
            partials[int64_t(blockIdx.x) * 3 + threadIdx.x] += v;
        }
    }
}

}  // namespace qlga
