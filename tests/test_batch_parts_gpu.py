"""Batch observables over runs of every length, split into parts or not, against the oracle, and their time on many
short runs: no more than 1.5 times that of a copy of the state and a wait, plus 120 us for every thousand runs (one CTA a
run takes 60 us a thousand; eight took 350).

Tolerance: 1e-6 of the norm in FP32, 1e-12 in FP64, as for the other read-outs.
"""
import ctypes
import time

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


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("lengths", [[8, 511, 512, 513, 2047, 2048, 2049, 9000], [40000], [100] * 700 + [5000]])
def test_parts(precision, lengths):
    rng = np.random.default_rng(len(lengths))
    dt = np.float32 if precision == 32 else np.float64
    states = [I.random_state(rng, n, scale=0.05).astype(dt) for n in lengths]
    b = qlga.Batch(lengths, [G] * len(lengths), precision=precision)
    b.load_state(np.concatenate([s.ravel() for s in states]))
    got = b.observables()
    b.close()
    tol = 1e-6 if precision == 32 else 1e-12
    for n, st, o in zip(lengths[::50] + lengths[-8:], states[::50] + states[-8:], got[::50] + got[-8:]):
        w = oracle.observables(np.ascontiguousarray(st, dtype=np.float64), oracle.make_cfg(1, n, 1, *G))
        for k in ("norm_qubit", "norm_boson", "magnetisation", "energy", "singlet_re", "singlet_im"):
            assert abs(o[k] - w[k]) <= tol * w["norm_qubit"], (n, k)


@pytest.mark.parametrize("nruns,L", [(4096, 64), (8192, 32)])
def test_many_short_runs(nruns, L):
    b = qlga.Batch([L] * nruns, [G] * nruns, precision=32)
    b.load_state(I.random_state(np.random.default_rng(1), nruns * L, scale=0.03).astype(np.float32).ravel())
    out, state = (qlga.QlgaObs * nruns)(), torch.empty(nruns * L * 20, device="cuda")
    lib, h = qlga.load_library(), ctypes.c_void_p(b.handle)

    def best(f):
        t = []
        for _ in range(10):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            f()
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t) * 1e6

    obs = best(lambda: qlga._check(lib.qlga_batch_observables(h, out), "observables"))
    get = best(lambda: qlga._check(lib.qlga_batch_get_state(h, ctypes.c_void_p(state.data_ptr()), qlga.QLGA_DEVICE), "get"))
    b.close()
    print("%d runs of %d: %.0f us, a copy %.0f" % (nruns, L, obs, get))
    assert obs <= 1.5 * get + 120.0 * nruns / 1000
