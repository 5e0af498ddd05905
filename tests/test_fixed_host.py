"""The integer fixed-point potential unitary on single sites, on the CPU: its functions compiled for the host
(fixed_host.cu) against the Taylor series of exp(-i delta V) in numpy's long double (at least 64 bits)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1907_12834_gb300 import build as qbuild

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
R = np.sqrt(np.longdouble(1.5))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fixed") / "fixed_host.so")
    cmd = [qbuild._nvcc(), "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
           "-Xcompiler", "-fPIC", "-shared", "-I", qbuild.CSRC, "-I", os.path.join(ROOT, "include"), "-o", so,
           os.path.join(HERE, "fixed_host.cu")]
    try:
        subprocess.run(cmd, check=True, capture_output=True, text=True)
    except FileNotFoundError:
        pytest.skip("nvcc not found")
    lib = ctypes.CDLL(so)
    lib.host_shift.restype = ctypes.c_longlong
    lib.host_shift.argtypes = [ctypes.c_longlong, ctypes.c_int]
    lib.host_density.restype = ctypes.c_double
    lib.host_density.argtypes = [ctypes.c_void_p]
    lib.host_potential.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double]
    return lib


def potential(lib, x, g, delta=1.0):
    """x (n, 5, 2) complex: U on every site in fixed point, and which sites are in its domain."""
    y = np.ascontiguousarray(x, dtype=np.complex128).copy()
    g = np.array(g, dtype=np.float64)
    ok = [lib.host_potential(s.ctypes.data, g.ctypes.data, delta) for s in y]
    return y, np.array(ok, dtype=bool)


def forms(p):
    """rho, F_z, F_+ of fields p (n, 5)."""
    n = p.real ** 2 + p.imag ** 2
    fz = 2 * (n[:, 0] - n[:, 4]) + n[:, 1] - n[:, 3]
    fp = 2 * (p[:, 0].conj() * p[:, 1] + p[:, 3].conj() * p[:, 4] + R * (p[:, 1].conj() * p[:, 2] + p[:, 2].conj() * p[:, 3]))
    return n.sum(axis=1), fz, fp


def reference(x, g, delta=1.0, dtype=np.clongdouble):
    """U by its Taylor series about V's centre, in the arithmetic of dtype."""
    real = np.zeros(1, dtype).real.dtype.type
    x = x.astype(dtype)
    p = x[:, :, 0] + x[:, :, 1]
    rho, fz, fp = forms(p)
    fz, fp = fz.astype(real), fp.astype(dtype)
    g0, g1, g2 = (real(v) * real(delta) for v in g)
    u = np.stack([p[:, 4], -p[:, 3], p[:, 2], -p[:, 1], p[:, 0]], axis=1)
    c = [real(1), real(R), real(R), real(1)]

    def w(v):  # (V - (g0 + g2 / 10) rho) v
        dot = (u * v).sum(axis=1)
        y = np.empty_like(v)
        for m in range(5):
            y[:, m] = (real(2 - m) * g1 * fz - g2 / 10 * rho) * v[:, m] + (g2 / 5) * u[:, m].conj() * dot
            if m < 4:
                y[:, m] += g1 * c[m] * fp.conj() * v[:, m + 1]
            if m > 0:
                y[:, m] += g1 * c[m - 1] * fp * v[:, m - 1]
        return y

    out = np.empty_like(x)
    theta = (g0 + g2 / 10) * rho
    phase = np.cos(theta) - 1j * np.sin(theta)
    for q in range(2):
        v = x[:, :, q].copy()
        for k in range(28, 0, -1):
            v = x[:, :, q] - dtype(1j) / real(k) * w(v)
        out[:, :, q] = phase[:, None] * v
    return out


def sites(rng, n, scale=0.05):
    return scale * (rng.standard_normal((n, 5, 2)) + 1j * rng.standard_normal((n, 5, 2)))


def test_shift_at_the_ends_of_its_domain(lib):
    """v 2^-n rounded to nearest for every n and |v| < 2^(58 + n), 2^62: the sum with the rounding bit may not wrap."""
    for n in range(-57, 6):
        top = (1 << min(58 + n, 62)) - 1
        for v in {top, top - 1, top // 2 + 1, 1, 0}:
            want = v << -n if n <= 0 else (v + (1 << (n - 1))) >> n
            assert lib.host_shift(v, n) == want, (v, n)
            assert abs(lib.host_shift(-v, n) + want) <= (n > 0)  # a half rounds up


def test_a_component_just_below_a_power_of_two(lib):
    """a + b = 2^59 - 1 units in the site's largest component: its rounding must not turn psi's sign.  Tolerance 4e-14
    of the site, as the domain test on the GPU."""
    g = (0.02, 0.02, 0.02)
    x = sites(np.random.default_rng(1), 2, 0.2)
    x[:, 2, 0] = 1.0 + 0.1j
    x[:, 2, 1] = -2.0 ** -59
    x[1] = -x[1]
    got, ok = potential(lib, x, g)
    ref = reference(x, g)
    assert ok.all()
    assert np.abs(got - ref).max() <= 4e-14 * np.abs(ref).max()


def test_density_is_not_biased(lib):
    """The mean relative error of rho over random sites: the dropped part of a square always has one sign and shifts
    every site's phase alike.  Tolerance 2^-55: four means' deviations of a sum rounded at 2^-53 over 4000 sites are
    below 2^-56, and the conversion to double that the test itself makes has none."""
    x = sites(np.random.default_rng(5), 4000)
    p = np.ascontiguousarray(x.sum(axis=2))
    got = np.array([lib.host_density(s.ctypes.data) for s in p])
    rho, _, _ = forms(p.astype(np.clongdouble))
    err = ((got - rho) / rho).astype(np.float64)
    assert abs(err.mean()) <= 2.0 ** -55, err.mean()


@pytest.mark.parametrize("g", [(1.0, 0.0, 0.0), (1.0, 0.1, 1.0), (0.0, 0.8, -0.6)])
def test_sites_of_one_density_share_no_phase(lib, g):
    """The mean phase of U's error over 400 sites of one density: a rounding of the phase or of W's diagonal that sites
    share would add up over a run's steps.  Tolerance 1.2e-17: the couplings' own rounding, up to four products of 2^-54
    of themselves at theta and beta below 0.03 (7e-18), and twice the mean's scatter (2^-54 / sqrt(4000))."""
    rng = np.random.default_rng(17)
    for rho in np.exp(rng.uniform(np.log(0.002), np.log(0.02), 12)):
        x = sites(rng, 400)
        p = x.sum(axis=2, keepdims=True)
        x = (0.5 * p + 0.25 * (x - x[:, :, ::-1])) * np.sqrt(rho / (np.abs(p) ** 2).sum(axis=(1, 2), keepdims=True))
        got, ok = potential(lib, x, g)
        ref = reference(x, g)
        assert ok.all()
        phase = float((ref.conj() * (got - ref)).imag.sum() / (np.abs(ref) ** 2).sum())
        assert abs(phase) <= 1.2e-17, (rho, phase)


def reached(x, g):
    """What reaches each level in U: |x_m| + sum_j |V_mj| |x_j| with the moduli's sums in V."""
    p, a = np.abs(x[:, :, 0] + x[:, :, 1]), np.abs(x).sum(axis=2)
    c = [1.0, 1.5 ** 0.5, 1.5 ** 0.5, 1.0]
    rho = (p ** 2).sum(axis=1, keepdims=True)
    fp = 2 * sum(c[i] * p[:, i] * p[:, i + 1] for i in range(4))
    out = a * (1 + (abs(g[0]) + 4 * abs(g[1]) + abs(g[2])) * rho) + abs(g[2]) / 5 * p[:, ::-1] * (p[:, ::-1] * a).sum(axis=1, keepdims=True)
    for m in range(4):
        out[:, m] += abs(g[1]) * c[m] * fp * a[:, m + 1]
        out[:, m + 1] += abs(g[1]) * c[m] * fp * a[:, m]
    return out


@pytest.mark.parametrize("g", [(1.0, 0.1, 1.0), (1.0, 0.8, -0.6)])
@pytest.mark.parametrize("kind,scale", [("plain", 0.002), ("plain", 0.02), ("plain", 0.05), ("polar", 1e-3), ("polar", 1e-10), ("polar", 1e-40),
                                        ("ends", 1e-6), ("ends", 1e-100), ("chain", 1e-3), ("chain", 1e-20), ("difference", 1e-6)])
def test_levels_are_as_exact_as_in_fp64(lib, kind, scale, g):
    """Each level's error over 400 sites, of what reaches it, no larger than that of the same series in FP64 (root mean
    square, with 10% for the scatter of 4000 numbers), and nowhere above 4 roundings of 2^-53."""
    rng = np.random.default_rng(23)
    x = sites(rng, 400, scale if kind == "plain" else 0.04)
    power = {"polar": (1, 1, 0, 1, 1), "ends": (0, 1, 1, 1, 0), "chain": (0, 1, 2, 3, 4)}.get(kind)
    if power:
        x = x * (scale ** np.array(power, dtype=float))[None, :, None]
    if kind == "difference":
        mean, diff = x.mean(axis=2, keepdims=True), (x - x[:, :, ::-1]) / 2
        x = mean * scale ** rng.uniform(0, 1, (400, 1, 1)) + diff * scale ** rng.uniform(0, 1, (400, 1, 1))
    got, ok = potential(lib, x, g)
    ref, f64, size = reference(x, g), reference(x, g, dtype=np.complex128), reached(x, g)[:, :, None]
    assert ok.all()
    err, err64 = ((np.abs(v - ref) / size).astype(np.float64) * 2.0 ** 53 for v in (got, f64))
    rms, rms64 = (np.sqrt((v ** 2).mean(axis=(0, 2))) for v in (err, err64))
    assert np.all(rms <= 1.1 * rms64) and err.max() <= 4.0, (rms, rms64, err.max())


def test_empty_levels_and_the_ends_of_the_domain(lib):
    """Empty sites and levels stay empty where nothing drives them; sites outside the domain are left alone."""
    rng = np.random.default_rng(2)
    x = sites(rng, 8, 0.04)
    x[0] = 0.0
    x[1, [0, 1, 3, 4]] = 0.0
    x[2, :, 0] = -x[2, :, 1]       # no field, only a difference
    x[3] *= 1e-250
    x[4, 3] *= 1e-300              # below the smallest level
    x[5] *= 20.0                   # a norm far above 1
    x[6, 2, 0] = np.inf
    x[7, 2, 0] = np.nan
    got, ok = potential(lib, x, (1.0, 0.8, -0.6))
    assert ok.tolist() == [True, True, True, True, False, False, False, False]
    same = x[4:]
    assert np.array_equal(got[4:], same, equal_nan=True)
    assert not got[0].any() and not got[1, [0, 1, 3, 4]].any()
    assert np.abs(got[2] - x[2]).max() <= 2.0 ** -53 * np.abs(x[2]).max()
    assert np.abs(got[3] - x[3]).max() <= 2.0 ** -53 * np.abs(x[3]).max()
