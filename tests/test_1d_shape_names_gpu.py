"""A 1D lattice's reported launch shape can be set on another lattice and gives it the same kernels; the shapes of four and
eight steps per launch, forced, on lattices of the widths where their tiles (100 and 72 sites) end.

Tolerances: 2e-5 of the norm in FP32, as the other forced shapes; the same bits for the same shape in FP64.
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


@pytest.mark.parametrize("steps", [4, 8])
@pytest.mark.parametrize("L", [8, 72, 73, 100, 104, 105, 1000])
@pytest.mark.parametrize("graph_steps", [0, 6, 32])
def test_four_and_eight_steps_per_launch(steps, L, graph_steps):
    st = I.random_state(np.random.default_rng(L), L, scale=0.03).astype(np.float32)
    n = 2 * graph_steps + 8 + 3
    ref = np.ascontiguousarray(st, dtype=np.float64)
    oracle.step(ref, oracle.make_cfg(1, L, 1, *G), n)
    with qlga.Lattice(1, L, precision=32, g=G) as lat:
        lat.set_1d_shape(128, 1, steps)
        lat.set_graph_steps(graph_steps)
        lat.load_state(st)
        lat.step(n)
        assert lat.shape_1d() == (128, 1, steps)
        got = lat.get_state()
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("precision,L", [(32, 1024), (32, 16384), (64, 1024), (64, 16384), (64, 33001)])
def test_reported_shape_is_accepted(precision, L):
    st = I.random_state(np.random.default_rng(L), L, scale=0.03).astype(np.float32 if precision == 32 else np.float64)
    shapes, states = [], []
    for shape in (None, "reported"):
        with qlga.Lattice(1, L, precision=precision, g=G) as lat:
            if shape:
                lat.set_1d_shape(*shapes[0])
            lat.load_state(st)
            lat.step(40)
            shapes.append(lat.shape_1d())
            states.append(lat.get_state())
    assert shapes[0] == shapes[1]
    if precision == 64:
        assert np.array_equal(states[0], states[1])


def test_where_several_steps_are_refused():
    for kw in ({"precision": 64}, {"precision": 32, "interleave": 1}):
        for steps in (4, 8):
            with qlga.Lattice(1, 300, g=G, **kw) as lat:
                with pytest.raises(qlga.QlgaError) as e:
                    lat.set_1d_shape(128, 1, steps)
                assert e.value.status == qlga.QLGA_ERR_UNSUPPORTED
    b = qlga.Batch([100, 64], [G] * 2, precision=32)
    with pytest.raises(qlga.QlgaError) as e:
        b.set_shape(128, 1, 4)
    b.close()
    assert e.value.status == qlga.QLGA_ERR_INVALID_ARG
