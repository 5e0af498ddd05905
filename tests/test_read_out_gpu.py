"""States read into a device buffer straight from K, and runs that take several steps per launch.

The direct read-out must give the bytes of the converted one (taken when the buffer is not 16-byte aligned):
the same arithmetic, only the layout of the store differs.  Runs of every length around the launches of
four and eight steps: 2e-5 of the norm against the oracle, as the 1D FP32 parity tests.
"""
import ctypes

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


@pytest.mark.parametrize("ndim,nx,ny", [(1, 131, 1), (1, 8, 1), (2, 64, 24), (2, 45, 19), (2, 20, 16), (2, 1024, 1030)])
@pytest.mark.parametrize("precision,variant", [(64, 0), (32, 0), (32, 1), (64, 1)])
def test_direct_read_out(ndim, nx, ny, precision, variant):
    dt = torch.float32 if precision == 32 else torch.float64
    st = I.random_state(np.random.default_rng(nx), nx, ny, scale=0.05)
    with qlga.Lattice(ndim, nx, ny, precision=precision, g=G, kinetic_variant=variant) as lat:
        lat.load_state(torch.tensor(st, dtype=dt, device="cuda"))
        lat.step(3)
        direct = lat.device_state()
        buf = torch.empty(direct.numel() + 1, dtype=dt, device="cuda")
        qlga.qlga_get_state(lat.handle, buf.data_ptr() + buf.element_size(), qlga.QLGA_DEVICE)
        lat.stream.synchronize()
        host = lat.get_state()
        again = lat.device_state()
    assert torch.equal(buf[1:], direct.reshape(-1)) and torch.equal(again, direct)
    assert np.array_equal(host, direct.cpu().numpy())


@pytest.mark.parametrize("precision,heights", [(32, None), (64, None), (32, [1, 40, 1])])
def test_batch_direct_read_out(precision, heights):
    lengths = [100, 64, 37]
    dt = torch.float32 if precision == 32 else torch.float64
    rng = np.random.default_rng(5)
    flat = np.concatenate([I.random_state(rng, n, h, scale=0.05).ravel() for n, h in zip(lengths, heights or [1] * 3)])
    b = qlga.Batch(lengths, [G] * 3, precision=precision, heights=heights)
    b.load_state(flat)
    b.step(5)
    bufs = []
    for off in (0, 1):
        t = torch.empty(flat.size + off, dtype=dt, device="cuda")
        qlga._check(qlga.load_library().qlga_batch_get_state(ctypes.c_void_p(b.handle), ctypes.c_void_p(t.data_ptr() + off * t.element_size()),
                                                             qlga.QLGA_DEVICE), "get")
        b.stream.synchronize()
        bufs.append(t[off:])
    host = b.get_state()
    b.close()
    assert torch.equal(bufs[0], bufs[1]) and np.array_equal(host, bufs[0].cpu().numpy())


@pytest.mark.parametrize("L", [8, 40, 104, 105, 1000, 16384])
@pytest.mark.parametrize("n,graph_steps", [(7, 32), (67, 32), (45, 34), (41, 6), (37, 0)])
def test_several_steps_per_launch(L, n, graph_steps):
    st = I.random_state(np.random.default_rng(L + n), L, scale=0.03).astype(np.float32)
    ref = np.ascontiguousarray(st, dtype=np.float64)
    oracle.step(ref, oracle.make_cfg(1, L, 1, *G), n)
    with qlga.Lattice(1, L, precision=32, g=G) as lat:
        qlga.qlga_set_graph_steps(lat.handle, graph_steps)
        lat.load_state(st)
        lat.step(n)
        o = lat.observables()
        got = lat.get_state()
    assert o["step"] == n
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)
