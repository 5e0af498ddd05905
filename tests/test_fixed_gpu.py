"""The integer fixed-point forms of the FP64 potential and of the 2D FP64 kinetic operator against the
oracle, at the edges of their domain.

Tolerances.  U: per site, 4e-14 of the site's norm (the fixed-point sums carry 2^-55 of it; the
oracle's Jacobi route to U about 30 units of 2^-53, ten times that allowed).  K: 2e-15 of the largest
component (one rounding of 2^-55 of the strip's largest between the axes, amplified by at most 44/16,
twice, and the conversions).
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


def _sites(kind, rng, nx):
    st = I.random_state(rng, nx, scale=0.05)
    if kind == "levels":      # levels of a site orders of magnitude apart, some empty
        st *= 10.0 ** rng.uniform(-9, 0, size=(5, 1, nx, 1, 1))
        st[rng.integers(0, 5, nx // 4), :, rng.integers(0, nx, nx // 4)] = 0.0
    elif kind == "tails":     # sites of one warp from 1e-250 to 1, and empty ones
        st *= 10.0 ** rng.uniform(-250, 0, size=(1, 1, nx, 1, 1))
        st[:, :, ::7] = 0.0
    elif kind == "difference":  # |a - b| far above |a + b|, and the other way round
        m = 0.5 * (st[..., 0, :] + st[..., 1, :]) * 10.0 ** rng.uniform(-6, 0, size=(1, 1, nx, 1))
        d = 0.5 * (st[..., 0, :] - st[..., 1, :]) * 10.0 ** rng.uniform(-6, 0, size=(1, 1, nx, 1))
        st[..., 0, :], st[..., 1, :] = m + d, m - d
    elif kind == "dense":     # sites beyond the fixed-point domain among the others of a warp
        st[:, :, rng.integers(0, nx, 5)] *= 4.0
    return st


@pytest.mark.parametrize("kind,g", [("plain", (1.0, -0.5, 0.2)), ("levels", (1.0, 0.8, -0.6)), ("tails", (1.0, 0.1, 1.0)),
                                    ("difference", (0.5, 0.3, 2.0)), ("dense", (1.0, 0.8, -0.6)),
                                    ("plain", (40.0, 0.1, 1.0)), ("plain", (0.0, 0.0, 0.0)), ("plain", (1.0, 0.0, 3.0))])
def test_potential_domain(kind, g):
    nx = 3 * 256 + 37
    rng = np.random.default_rng(len(kind) + int(10 * g[0]))
    st = _sites(kind, rng, nx)
    ref = np.ascontiguousarray(st).copy()
    oracle.apply_potential(ref, oracle.make_cfg(1, nx, 1, *g), 1.0)
    with qlga.Lattice(1, nx, precision=64, g=g) as lat:
        lat.load_state(st)
        lat.apply_potential(1.0)
        got = lat.get_state()
    err = np.sqrt(((got - ref) ** 2).sum(axis=(0, 1, 3, 4)))
    norm = np.sqrt((ref ** 2).sum(axis=(0, 1, 3, 4)))
    assert np.all(err <= 4e-14 * norm), float(np.max(err / np.maximum(norm, 1e-300)))


@pytest.mark.parametrize("nx,ny,variant", [(32, 8, 0), (33, 9, 1), (63, 21, 0), (64, 8, 1), (95, 40, 0), (256, 67, 1)])
@pytest.mark.parametrize("rows", ["even", "jumps"])
def test_kinetic_strips(nx, ny, variant, rows):
    rng = np.random.default_rng(nx + ny)
    st = I.random_state(rng, nx, ny, scale=0.05)
    if rows == "jumps":       # the pipeline's exponent rises and falls along y
        st *= 2.0 ** rng.integers(-40, 1, size=(1, ny, 1, 1, 1))
    ref = np.ascontiguousarray(st).copy()
    oracle.step(ref, oracle.make_cfg(2, nx, ny, 0.0, 0.0, 0.0, kinetic_variant=variant), 2)
    with qlga.Lattice(2, nx, ny, precision=64, g=(0.0, 0.0, 0.0), kinetic_variant=variant) as lat:
        lat.load_state(st)
        lat.step(2)
        got = lat.get_state()
    assert np.abs(got - ref).max() <= 2e-15 * np.abs(ref).max()


def test_nan_in_a_strip_is_reported():
    st = I.random_state(np.random.default_rng(3), 70, 20, scale=0.05)
    st[2, 11, 40, 1, 0] = np.nan
    with qlga.Lattice(2, 70, 20, precision=64, g=(1.0, 0.1, 1.0)) as lat:
        lat.load_state(st)
        with pytest.raises(qlga.QlgaError) as ei:
            lat.step(3)
            lat.get_state()
        assert ei.value.status == qlga.QLGA_ERR_NOT_FINITE
