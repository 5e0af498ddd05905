"""The fixed-point pull-back of an FP64 step against the oracle's, at the edges of its domain: levels and sites
orders of magnitude apart, empty sites and cotangents, |a - b| far from |a + b|, sites that leave the domain (their warps
take the FP64 code), large phases, and no couplings.

Tolerance: that of one step in test_adjoint_gpu.py, 1e-11 of the norm of the cotangent's pull-back, and of the
largest coupling gradient.
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


@pytest.mark.parametrize("kind,g", [("plain", (1.0, -0.5, 0.2)), ("levels", (1.0, 0.8, -0.6)), ("tails", (1.0, 0.1, 1.0)),
                                    ("difference", (0.5, 0.3, 2.0)), ("dense", (1.0, 0.8, -0.6)), ("plain", (40.0, 0.1, 1.0)),
                                    ("plain", (0.0, 0.0, 0.0)), ("plain", (1.0, 0.0, 3.0)), ("cotangents", (1.0, 0.1, 1.0))])
@pytest.mark.parametrize("nx,ny", [(150, 1), (37, 12)])
def test_pull_back_domain(kind, g, nx, ny):
    rng = np.random.default_rng(nx + len(kind))
    st = I.random_state(rng, nx, ny, scale=0.05)
    cot = rng.standard_normal(st.shape)
    if kind == "levels":
        st *= 10.0 ** rng.uniform(-9, 0, size=(5, ny, nx, 1, 1))
        st[rng.integers(0, 5, nx // 4), :, rng.integers(0, nx, nx // 4)] = 0.0
    elif kind == "tails":
        st *= 10.0 ** rng.uniform(-120, 0, size=(1, ny, nx, 1, 1))
        st[:, :, ::7] = 0.0
    elif kind == "difference":
        m = 0.5 * (st[..., 0, :] + st[..., 1, :]) * 10.0 ** rng.uniform(-6, 0, size=(1, ny, nx, 1))
        d = 0.5 * (st[..., 0, :] - st[..., 1, :]) * 10.0 ** rng.uniform(-6, 0, size=(1, ny, nx, 1))
        st[..., 0, :], st[..., 1, :] = m + d, m - d
    elif kind == "dense":
        st[:, :, rng.integers(0, nx, 2)] *= 2.5
    elif kind == "cotangents":
        cot *= 10.0 ** rng.uniform(-200, 60, size=(1, ny, nx, 1, 1))
        cot[:, :, ::3] = 0.0
    ndim = 1 if ny == 1 else 2
    ref = cot.copy()
    dref = oracle.vjp_step(np.ascontiguousarray(st), ref, oracle.make_cfg(ndim, nx, ny, *g))
    with qlga.Lattice(ndim, nx, ny, precision=64, g=g) as lat:
        got, dg = lat.adjoint_step(torch.tensor(st, device="cuda"), torch.tensor(cot, device="cuda"))
    assert np.linalg.norm(got.cpu().numpy() - ref) <= 1e-11 * np.linalg.norm(ref)
    assert np.abs(dg - dref).max() <= 1e-11 * max(np.abs(dref).max(), np.abs(cot).max() * np.abs(st).max() ** 3)


# K^dagger alone (no couplings), at the ends of strips and chunks: 2e-15 of the largest component (one rounding of 2^-54 of the
# strip's largest between the axes, amplified by at most 44/16, twice, and the conversions)
@pytest.mark.parametrize("nx,ny,variant", [(32, 8, 0), (33, 9, 1), (63, 21, 0), (64, 8, 1), (95, 40, 0), (256, 67, 1), (31, 12, 0)])
@pytest.mark.parametrize("rows", ["even", "jumps"])
def test_kinetic_adjoint_strips(nx, ny, variant, rows):
    rng = np.random.default_rng(nx + ny)
    st = I.random_state(rng, nx, ny, scale=0.05)
    cot = rng.standard_normal(st.shape)
    if rows == "jumps":
        cot *= 2.0 ** rng.integers(-40, 1, size=(1, ny, 1, 1, 1))
    ref = cot.copy()
    oracle.vjp_step(np.ascontiguousarray(st), ref, oracle.make_cfg(2, nx, ny, 0.0, 0.0, 0.0, kinetic_variant=variant))
    with qlga.Lattice(2, nx, ny, precision=64, g=(0.0, 0.0, 0.0), kinetic_variant=variant) as lat:
        got, _ = lat.adjoint_step(torch.tensor(st, device="cuda"), torch.tensor(cot, device="cuda"))
    assert np.abs(got.cpu().numpy() - ref).max() <= 2e-15 * np.abs(ref).max()


def test_nan_cotangent_stays_visible():
    nx, ny = 70, 20
    rng = np.random.default_rng(4)
    st, cot = I.random_state(rng, nx, ny, scale=0.05), rng.standard_normal((5, ny, nx, 2, 2))
    cot[1, 9, 40, 0, 1] = np.nan
    with qlga.Lattice(2, nx, ny, precision=64, g=(1.0, 0.1, 1.0)) as lat:
        got, dg = lat.adjoint_step(torch.tensor(st, device="cuda"), torch.tensor(cot, device="cuda"))
    assert np.isnan(got[:, 9, 40].cpu().numpy()).any() and np.isnan(dg).any()
