"""A step launched by itself costs the host no more than its kernels take: narrow lattices of many rows, whose split into
row chunks is searched for once per lattice.  Time per step without a step graph at most 1.33 times that within one (the gap of
a launch is 3 us of 13)."""
import numpy as np
import pytest

from paper_1907_12834_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1907_12834_gb300 import qlga  # noqa: E402


@pytest.mark.parametrize("nx,ny", [(32, 4096), (96, 1300)])
def test_single_steps_of_narrow_lattices(nx, ny):
    st = I.random_state(np.random.default_rng(1), nx, ny, scale=0.03).astype(np.float32)
    us = {}
    for graph_steps in (32, 0):
        with qlga.Lattice(2, nx, ny, precision=32, g=(1.0, 0.1, 1.0)) as lat:
            lat.set_graph_steps(graph_steps)
            lat.load_state(st)
            lat.step(66)
            best = np.inf
            for _ in range(6):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                e0.record(lat.stream)
                lat.step(320)
                e1.record(lat.stream)
                torch.cuda.synchronize()
                best = min(best, e0.elapsed_time(e1) * 1e3 / 320)
            us[graph_steps] = best
    print("%d x %d: %.2f us a step, %.2f in a graph" % (nx, ny, us[0], us[32]))
    assert us[0] <= 1.33 * us[32]
