"""The kernels that march down rows with one strip of columns per warp, at the edges of their strips and
chunks, against the oracle: fields and observables of a true 2D state, the FP32 step by levels, and the
interleaved step's y pass by tiles.  Tolerances: those of the same quantities in test_parity_gpu.py.
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

G = (1.0, 0.8, -0.6)


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nx,ny", [(8, 9), (29, 8), (30, 16), (31, 17), (32, 33), (61, 40), (65, 23)])
def test_fields_and_observables_of_a_true_state(precision, nx, ny):
    rng = np.random.default_rng(nx * ny + precision)
    dt = np.float32 if precision == 32 else np.float64
    st, ref_st = (I.random_state(rng, nx, ny, scale=0.1).astype(dt) for _ in range(2))
    cfg = oracle.make_cfg(2, nx, ny, *G)
    with qlga.Lattice(2, nx, ny, precision=precision, g=G) as lat:
        lat.load_state(st)
        got = lat.fields()
        o = lat.observables(ref=torch.from_numpy(ref_st).cuda())
        parts = [lat.observable_sums(a, b) for a, b in ((0, ny // 3), (ny // 3, ny))]
        whole = lat.observable_sums()
    st64 = np.ascontiguousarray(st, dtype=np.float64)
    ref = oracle.fields(st64, cfg)
    scale = np.abs(ref[:3]).max()
    np.testing.assert_allclose(got[:3], ref[:3], rtol=0, atol=(1e-12 if precision == 64 else 2e-5) * scale)
    np.testing.assert_allclose(got[6:], ref[6:], rtol=0, atol=1e-9 if precision == 64 else 1e-6)
    w = oracle.observables(st64, cfg, ref=np.ascontiguousarray(ref_st, dtype=np.float64))
    tol = 1e-6 if precision == 32 else 1e-12
    for k in ("norm_qubit", "norm_boson", "magnetisation", "energy", "singlet_re", "singlet_im", "overlap_re", "overlap_im"):
        assert abs(o[k] - w[k]) <= tol * w["norm_qubit"], k
    np.testing.assert_allclose(parts[0] + parts[1], whole, rtol=0, atol=tol * w["norm_qubit"])


# both sides of the line between the step by levels and by strips (2^17 sites), rows in and out of fives
@pytest.mark.parametrize("nx,ny", [(32, 8), (64, 13), (96, 40), (131, 9), (256, 511), (256, 513), (363, 362)])
@pytest.mark.parametrize("variant", [0, 1])
def test_step_by_levels(nx, ny, variant):
    rng = np.random.default_rng(nx + 3 * ny)
    st = I.random_state(rng, nx, ny, scale=0.05).astype(np.float32)
    ref = np.ascontiguousarray(st, dtype=np.float64)
    oracle.step(ref, oracle.make_cfg(2, nx, ny, *G, kinetic_variant=variant), 7)
    with qlga.Lattice(2, nx, ny, precision=32, g=G, kinetic_variant=variant) as lat:
        lat.load_state(st)
        lat.step(7)
        got = lat.get_state()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("nx,ny", [(8, 8), (33, 56), (62, 57), (101, 112), (130, 130)])
@pytest.mark.parametrize("precision", [64, 32])
def test_interleaved_tiles(nx, ny, precision):
    rng = np.random.default_rng(nx + ny)
    st = I.random_state(rng, nx, ny, scale=0.05).astype(np.float32 if precision == 32 else np.float64)
    ref = np.ascontiguousarray(st, dtype=np.float64).copy()
    oracle.step(ref, oracle.make_cfg(2, nx, ny, *G, interleave=1), 4)
    with qlga.Lattice(2, nx, ny, precision=precision, g=G, interleave=1) as lat:
        lat.load_state(st)
        lat.step(4)
        got = lat.get_state()
    assert np.linalg.norm(got - ref) <= (1e-11 if precision == 64 else 1e-5) * np.linalg.norm(ref)


@pytest.mark.parametrize("nx,ny", [(96, 70), (101, 64)])
@pytest.mark.parametrize("variant", [0, 1])
def test_tails_of_a_localised_fp64_state(nx, ny, variant):
    """K of a 2D FP64 state runs on integers with one exponent per strip of 40 columns and 16 rows; strips with a column
    2^-20 below the largest take FP64.  Every site within 1e-9 of the largest within the 8 rows and columns that two
    steps reach (2^-54 of a strip's largest is 2^-34 of its smallest column, amplified by at most (44/16)^2 a
    step)."""
    rng = np.random.default_rng(nx)
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    env = np.exp(-1.1 * np.sqrt((x - nx / 2.0) ** 2 + (y - ny / 2.0) ** 2))
    st = I.random_state(rng, nx, ny, scale=0.05) * env[None, :, :, None, None]
    ref = np.ascontiguousarray(st).copy()
    oracle.step(ref, oracle.make_cfg(2, nx, ny, *G, kinetic_variant=variant), 2)
    with qlga.Lattice(2, nx, ny, precision=64, g=G, kinetic_variant=variant) as lat:
        lat.load_state(st)
        lat.step(2)
        got = lat.get_state()
    err = np.sqrt(((got - ref) ** 2).sum(axis=(0, 3, 4)))
    near = np.sqrt((st ** 2).sum(axis=(0, 3, 4)))
    for axis in (0, 1):
        near = np.max([np.roll(near, k, axis=axis) for k in range(-8, 9)], axis=0)
    assert np.all(err <= 1e-9 * near), float(np.max(err / near))
