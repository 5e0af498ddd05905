"""The fixed-point FP64 step of a 1D lattice against the oracle: ten, five and one lane per site (chosen by the
length), at the ends of a warp's sites, on lattices shorter than a warp's columns, and on states whose
sites lie far apart in size.

Tolerance: 1e-13 of the largest site within the 24 sites that three steps and the read-out reach (the
integer sums resolve 2^-51 of the largest of nine columns, four roundings a step; the oracle's Jacobi
route to U is good to about 30 units of 2^-53).
"""
import numpy as np
import pytest

import oracle
from paper_1907_12834_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1907_12834_gb300 import qlga  # noqa: E402


def _state(kind, rng, L):
    st = I.random_state(rng, L, scale=0.05)
    if kind == "tail":      # a site 2^-40 of its neighbour's neighbour and less, down to nothing
        x = np.arange(L)
        st *= np.exp(-1.7 * np.minimum(x, L - x)).reshape(1, 1, L, 1, 1)
        st[:, :, L // 2:L // 2 + 3] = 0.0
    elif kind == "islands":  # empty but for a few sites
        keep = np.zeros(L)
        keep[rng.integers(0, L, max(1, L // 40))] = 1.0
        st *= keep.reshape(1, 1, L, 1, 1)
    elif kind == "dense":   # some warps leave the fixed-point domain
        st[:, :, rng.integers(0, L, max(1, L // 200))] *= 5.0
    return st


def _beta(st, g):
    """The largest bound of ||delta (V - c)|| over the sites, 2 |g1| |F| + |g2| rho / 10."""
    p = st[:, 0, :, 0] + st[:, 0, :, 1]
    p = p[..., 0] + 1j * p[..., 1]
    n = np.abs(p) ** 2
    fz = 2 * (n[0] - n[4]) + n[1] - n[3]
    fp = 2 * (p[0].conj() * p[1] + p[3].conj() * p[4] + np.sqrt(1.5) * (p[1].conj() * p[2] + p[2].conj() * p[3]))
    return float(np.max(2 * abs(g[1]) * np.sqrt(fz ** 2 + np.abs(fp) ** 2) + 0.1 * abs(g[2]) * n.sum(axis=0)))


@pytest.mark.parametrize("L,variant", [(8, 0), (31, 1), (32, 0), (61, 0), (100, 1), (4096, 0), (4097, 1), (9001, 0), (24001, 0), (24100, 1)])
@pytest.mark.parametrize("kind", ["plain", "tail", "islands", "dense"])
def test_steps(L, variant, kind):
    g = (1.0, 0.8, -0.6)
    st = _state(kind, np.random.default_rng(L + len(kind)), L)
    ref = np.ascontiguousarray(st).copy()
    oracle.step(ref, oracle.make_cfg(1, L, 1, *g, kinetic_variant=variant), 3)
    with qlga.Lattice(1, L, precision=64, g=g, kinetic_variant=variant) as lat:
        lat.load_state(st)
        lat.step(3)
        assert lat.shape_1d() == (32, 1, 1)
        if _beta(st, g) > 4.0:  # outside the step's range in any arithmetic
            with pytest.raises(qlga.QlgaError) as ei:
                lat.get_state()
            assert ei.value.status == qlga.QLGA_ERR_NOT_FINITE
            return
        got = lat.get_state()
    err = np.sqrt(((got - ref) ** 2).sum(axis=(0, 1, 3, 4)))
    size = np.maximum(np.sqrt((ref ** 2).sum(axis=(0, 1, 3, 4))), np.sqrt((st ** 2).sum(axis=(0, 1, 3, 4))))
    near = np.max([np.roll(size, k) for k in range(-24, 25)], axis=0)
    assert np.all(err <= 1e-13 * near), float(np.max(err / np.maximum(near, 1e-300)))


@pytest.mark.parametrize("L", [50, 5000, 30000])
def test_nan_is_reported(L):
    st = I.random_state(np.random.default_rng(3), L, scale=0.05)
    st[2, 0, L // 2, 1, 0] = np.nan
    with qlga.Lattice(1, L, precision=64, g=(1.0, 0.8, -0.6)) as lat:
        lat.load_state(st)
        with pytest.raises(qlga.QlgaError) as ei:
            lat.step(3)
            lat.get_state()
        assert ei.value.status == qlga.QLGA_ERR_NOT_FINITE
