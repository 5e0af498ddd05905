"""The potential unitary with a negative delta against the oracle, and a step forward after it.  The Taylor degree comes from beta = ||delta W||, which must not carry delta's sign.

Tolerances: 1e-13 of the norm in FP64 (the oracle's Jacobi route to U is good to about 30 units of 2^-53), 3e-6 in FP32 (terms up to e^beta = 9, 6e-8 each),
each twice that for the two steps.
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


@pytest.mark.parametrize("nx,ny", [(131, 1), (40, 24)])
@pytest.mark.parametrize("delta", [-0.5, -1.0, -5.0])
@pytest.mark.parametrize("precision,tol", [(64, 1e-13), (32, 3e-6)])
def test_step_back(nx, ny, delta, precision, tol):
    dt = np.float32 if precision == 32 else np.float64
    st = I.random_state(np.random.default_rng(nx), nx, ny, scale=0.05).astype(dt)
    ref = np.ascontiguousarray(st, dtype=np.float64).copy()
    ndim = 1 if ny == 1 else 2
    oracle.apply_potential(ref, oracle.make_cfg(ndim, nx, ny, *G), delta)
    with qlga.Lattice(ndim, nx, ny, precision=precision, g=G) as lat:
        lat.load_state(st)
        lat.apply_potential(delta)
        back = lat.get_state()
        lat.apply_potential(-delta)
        again = lat.get_state()
    assert np.linalg.norm(back - ref) <= tol * np.linalg.norm(ref)
    oracle.apply_potential(ref, oracle.make_cfg(ndim, nx, ny, *G), -delta)
    assert np.linalg.norm(again - ref) <= 2 * tol * np.linalg.norm(ref)


def test_a_large_negative_delta_is_reported_as_a_positive_one():
    st = I.random_state(np.random.default_rng(2), 64, 1, scale=0.05)
    for delta in (1e4, -1e4):
        for precision in (64, 32):
            with qlga.Lattice(1, 64, precision=precision, g=G) as lat:
                lat.load_state(st)
                with pytest.raises(qlga.QlgaError) as ei:
                    lat.apply_potential(delta)
                    lat.get_state()
                assert ei.value.status == qlga.QLGA_ERR_NOT_FINITE
