"""FP32 2D lattices a little wider than a strip of 32 columns: steps against the oracle on either side of the line between
two passes and strips, and the default no slower than two passes (10% for the timing's scatter)."""
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


# the last strip has one column, a few, or all but one; 2^17 sites between (97, 1351) and (97, 1352)
@pytest.mark.parametrize("nx,ny", [(33, 40), (65, 40), (66, 40), (97, 30), (129, 30), (129, 1100), (127, 9), (97, 1351), (97, 1352), (33, 31800)])
@pytest.mark.parametrize("variant", [0, 1])
def test_steps(nx, ny, variant):
    st = I.random_state(np.random.default_rng(nx + ny), nx, ny, scale=0.05).astype(np.float32)
    ref = np.ascontiguousarray(st, dtype=np.float64)
    n = 5 if nx * ny < 200000 else 2
    oracle.step(ref, oracle.make_cfg(2, nx, ny, *G, kinetic_variant=variant), n)
    with qlga.Lattice(2, nx, ny, precision=32, g=G, kinetic_variant=variant) as lat:
        lat.load_state(st)
        lat.step(n)
        o = lat.observables()
        got = lat.get_state()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
    w = oracle.observables(np.ascontiguousarray(got, dtype=np.float64), oracle.make_cfg(2, nx, ny, *G, kinetic_variant=variant))
    for k in ("norm_qubit", "norm_boson", "energy"):
        assert abs(o[k] - w[k]) <= 1e-6 * w["norm_qubit"], k


@pytest.mark.parametrize("nx,ny", [(33, 3030), (36, 2777), (40, 2500), (65, 1538), (34, 14705), (100, 1000), (1000, 701)])
def test_the_default_is_the_faster_form(nx, ny):
    st = I.random_state(np.random.default_rng(nx), nx, ny, scale=0.03).astype(np.float32)
    us = {}
    for mode in (qlga.QLGA_STEP2D_AUTO, qlga.QLGA_STEP2D_TWO_PASS):
        with qlga.Lattice(2, nx, ny, precision=32, g=(1.0, 0.1, 1.0)) as lat:
            lat.set_step2d_mode(mode)
            lat.load_state(st)
            lat.step(66)
            us[mode] = np.inf
            for _ in range(5):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(lat.stream)
                lat.step(32)
                e1.record(lat.stream)
                torch.cuda.synchronize()
                us[mode] = min(us[mode], e0.elapsed_time(e1) * 1e3 / 32)
    assert us[qlga.QLGA_STEP2D_AUTO] <= 1.1 * us[qlga.QLGA_STEP2D_TWO_PASS], us
