// Host library for tests/test_fixed_host.py: the integer fixed-point arithmetic of qlga_fixed.cuh on single sites.
// Built with nvcc for the host; no kernel is launched and no GPU is needed.
#include "qlga_device.cuh"

using namespace qlga;

extern "C" {

long long host_shift(long long v, int n) { return fx_scale(v, -n); }

// The density of a field psi[level][re, im]
double host_density(const double* psi) {
    FxLevels p;
    for (int i = 0; i < 5; ++i) {
        const int E = fx_exponent(fx_top(fx_top(0, psi[2 * i]), psi[2 * i + 1]));
        fx_level(fx_from_double<60>(psi[2 * i], E), fx_from_double<60>(psi[2 * i + 1], E), E - 1022 - 60, p.p.re[i], p.p.im[i], p.e[i]);
    }
    FxForms f;
    fx_forms(p, FixPot(0, 0, 0, 0, 0), f);
    return std::ldexp(double(f.rho), f.en - 56);
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
