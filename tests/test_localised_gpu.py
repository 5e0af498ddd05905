"""K and K^dagger of a localised 2D FP64 field: every site keeps the digits of its own neighbourhood, as FP64 does, wherever the
field within the kernel's strip of 40 columns and 16 rows varies.

Tolerance: 6e-15 of the largest component within reach (8 rows and columns for two steps).  An axis of K is 24 sums of
at most 16 times the input, divided by 16: up to four roundings of 2^-53 root mean square, so 24 for two axes, two steps and the
margin of a maximum, on either side (the oracle works in FP64 too).
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

TOL = 6e-15


def _envelope(kind, rng, nx, ny):
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    one = np.ones((ny, nx))
    if kind == "even":
        return one
    if kind == "tail x":
        return 2.0 ** -np.minimum(x, nx - x) * one
    if kind == "tail y":
        return 2.0 ** -np.minimum(y, ny - y) * one
    if kind == "tail":      # a soliton of the lattice scaling in both directions
        return np.exp(-0.1 * np.hypot(x - nx / 2, y - ny / 2))
    if kind == "island":    # full, then empty, then something small on the last four columns of a strip
        e = one.copy()
        e[:, 16:] = 0.0
        e[:, 28:32] = 1e-12
        return e
    if kind == "rows":
        return 2.0 ** rng.integers(-40, 1, size=(ny, 1)) * one
    if kind == "patches":   # eight by eight sites of a size each, some empty
        e = 10.0 ** rng.uniform(-30, 0, size=((ny + 7) // 8, (nx + 7) // 8))
        e[rng.random(e.shape) < 0.3] = 0.0
        return np.kron(e, np.ones((8, 8)))[:ny, :nx]
    raise ValueError(kind)


KINDS = ["even", "tail x", "tail y", "tail", "island", "rows", "patches"]


def _near(field, reach):
    size = np.abs(field).max(axis=(3, 4))  # (5, ny, nx)
    for axis in (1, 2):
        size = np.max([np.roll(size, k, axis=axis) for k in range(-reach, reach + 1)], axis=0)
    return size


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nx,ny,variant", [(96, 70, 0), (101, 64, 1), (40, 200, 0)])
def test_kinetic(kind, nx, ny, variant):
    rng = np.random.default_rng(nx + len(kind))
    st = I.random_state(rng, nx, ny, scale=0.05) * _envelope(kind, rng, nx, ny)[None, :, :, None, None]
    ref = np.ascontiguousarray(st).copy()
    oracle.step(ref, oracle.make_cfg(2, nx, ny, 0.0, 0.0, 0.0, kinetic_variant=variant), 2)
    with qlga.Lattice(2, nx, ny, precision=64, g=(0.0, 0.0, 0.0), kinetic_variant=variant) as lat:
        lat.load_state(st)
        lat.step(2)
        got = lat.get_state()
    err, near = np.abs(got - ref).max(axis=(3, 4)), _near(st, 8)
    assert np.all(err <= TOL * near), float((err / np.maximum(near, 1e-300)).max())


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nx,ny,variant", [(96, 70, 0), (101, 64, 1), (40, 200, 0)])
def test_kinetic_adjoint(kind, nx, ny, variant):
    rng = np.random.default_rng(nx + len(kind))
    st = I.random_state(rng, nx, ny, scale=0.05)
    cot = rng.standard_normal(st.shape) * _envelope(kind, rng, nx, ny)[None, :, :, None, None]
    ref = cot.copy()
    oracle.vjp_kinetic(ref, oracle.make_cfg(2, nx, ny, 0.0, 0.0, 0.0, kinetic_variant=variant))
    with qlga.Lattice(2, nx, ny, precision=64, g=(0.0, 0.0, 0.0), kinetic_variant=variant) as lat:
        got, _ = lat.adjoint_step(torch.tensor(st, device="cuda"), torch.tensor(cot, device="cuda"))
    err, near = np.abs(got.cpu().numpy() - ref).max(axis=(3, 4)), _near(cot, 4)
    assert np.all(err <= 0.5 * TOL * near), float((err / np.maximum(near, 1e-300)).max())


def _reach_of(bad, y, x):
    """Whether the sites that are not finite lie within K's reach of (y, x), and that one among them."""
    out = bad.copy()
    out[y - 4:y + 5, x - 4:x + 5] = False
    return bad[y, x] and not out.any()


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_what_is_not_finite_reaches_its_stencil_alone(value):
    nx, ny = 70, 40
    rng = np.random.default_rng(2)
    st, cot = I.random_state(rng, nx, ny, scale=0.05), rng.standard_normal((5, ny, nx, 2, 2))
    bad_st, bad_cot = st.copy(), cot.copy()
    bad_st[1, 20, 30, 0, 1] = bad_cot[1, 20, 30, 0, 1] = value
    with qlga.Lattice(2, nx, ny, precision=64, g=(1.0, 0.1, 1.0)) as lat:
        dev = torch.empty(st.shape, dtype=torch.float64, device="cuda")
        lat.load_state(torch.tensor(bad_st, device="cuda"))
        lat.step(1)
        got = lat.get_state(dev).cpu().numpy()
    assert _reach_of(~np.isfinite(got).all(axis=(0, 3, 4)), 20, 30)
    with qlga.Lattice(2, nx, ny, precision=64, g=(1.0, 0.1, 1.0)) as lat:
        got, _ = lat.adjoint_step(torch.tensor(st, device="cuda"), torch.tensor(bad_cot, device="cuda"))
    assert _reach_of(~np.isfinite(got.cpu().numpy()).all(axis=(0, 3, 4)), 20, 30)


def test_large_cotangents_are_pulled_back():
    nx, ny = 70, 40
    rng = np.random.default_rng(2)
    st, cot = I.random_state(rng, nx, ny, scale=0.05), rng.standard_normal((5, ny, nx, 2, 2))
    cot[1, 20:24, 30:34] *= 1e295
    ref = cot.copy()
    oracle.vjp_kinetic(ref, oracle.make_cfg(2, nx, ny, 0.0, 0.0, 0.0))
    with qlga.Lattice(2, nx, ny, precision=64, g=(0.0, 0.0, 0.0)) as lat:
        got, _ = lat.adjoint_step(torch.tensor(st, device="cuda"), torch.tensor(cot, device="cuda"))
    assert np.all(np.abs(got.cpu().numpy() - ref).max(axis=(3, 4)) <= 0.5 * TOL * _near(cot, 4))
