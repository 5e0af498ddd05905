// Host library for tests/test_fixed_host.py: the integer fixed-point arithmetic of qlga_fixed.cuh on single sites.
// Built with nvcc for the host; no kernel is launched and no GPU is needed.
#include "qlga_device.cuh"

using namespace qlga;

extern "C" {

long long host_shift(long long v, int n) { return fx_shift(v, n); }

// The density of a field psi[level][re, im]
double host_density(const double* psi) {
    unsigned m = 0;
    for (int i = 0; i < 10; ++i) m = fx_top(m, psi[i]);
    const int E = fx_exponent(m);
    i64 re[5], im[5];
    for (int i = 0; i < 5; ++i) {
        re[i] = fx_from_double<60>(psi[2 * i], E);
        im[i] = fx_from_double<60>(psi[2 * i + 1], E);
    }
    const int n = fx_headroom(re, im);
    FxVec p;
    for (int i = 0; i < 5; ++i) {
        p.re[i] = fx_split(fx_shift(re[i], n));
        p.im[i] = fx_split(fx_shift(im[i], n));
    }
    FxForms f;
    fx_forms(p, f);
    return std::ldexp(double(f.rho), 2 * (E - 1022 - 60 + n) + 60);
}

// U on the pair (a, b) of a site; x[level][qubit][re, im], in place.  Returns whether the site is in the domain.
int host_potential(double* x, const double* g, double delta) {
    const PotConst<double> C(PotParams{g[0], g[1], g[2], delta});
    double ar[5], ai[5], br[5], bi[5];
    for (int m = 0; m < 5; ++m) {
        ar[m] = x[4 * m];
        ai[m] = x[4 * m + 1];
        br[m] = x[4 * m + 2];
        bi[m] = x[4 * m + 3];
    }
    if (!fx_potential<false>(ar, ai, br, bi, 0, -1, C.fx)) return 0;
    for (int m = 0; m < 5; ++m) {
        x[4 * m] = ar[m];
        x[4 * m + 1] = ai[m];
        x[4 * m + 2] = br[m];
        x[4 * m + 3] = bi[m];
    }
    return 1;
}
}
