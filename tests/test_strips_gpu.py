"""The FP32 warp-strip step and observables read-out on widths that end inside a strip: steps against the
oracle, the read-out against the oracle's observables of the same state, and both against the two-pass form.

Tolerances: those of the fused step on multiples of 32 (steps 1e-5 relative L2; FP32 terms of the sums 1e-6 of
the norm, 2e-6 against the two-pass K, which rounds differently).
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


@pytest.mark.parametrize("nx,ny,variant", [(33, 8, 0), (33, 41, 1), (63, 9, 1), (65, 21, 0), (95, 40, 1), (250, 67, 0), (1000, 13, 0)])
def test_ragged_strips(nx, ny, variant):
    rng = np.random.default_rng(nx + ny)
    st = I.random_state(rng, nx, ny, scale=0.05).astype(np.float32)
    ref_st = I.random_state(rng, nx, ny, scale=0.05).astype(np.float32)
    ref_dev = torch.from_numpy(ref_st).cuda()
    cfg = oracle.make_cfg(2, nx, ny, *G, kinetic_variant=variant)
    with qlga.Lattice(2, nx, ny, precision=32, g=G, kinetic_variant=variant) as lat:
        lat.load_state(st)
        lat.step(12)
        o, o_again = lat.observables(ref=ref_dev), lat.observables(ref=ref_dev)
        got = lat.get_state()
        lat.set_step2d_mode(qlga.QLGA_STEP2D_TWO_PASS)
        o_two = lat.observables(ref=ref_dev)
        lat.load_state(st)
        lat.step(12)
        two = lat.get_state()
    ref = np.ascontiguousarray(st, dtype=np.float64)
    oracle.step(ref, cfg, 12)
    for x in (got, two):
        assert np.linalg.norm(x - ref) <= 1e-5 * np.linalg.norm(ref)
    w = oracle.observables(np.ascontiguousarray(got, dtype=np.float64), cfg, ref=np.ascontiguousarray(ref_st, dtype=np.float64))
    scale = w["norm_qubit"]
    for k in ("norm_qubit", "norm_boson", "magnetisation", "energy", "singlet_re", "singlet_im", "overlap_re", "overlap_im"):
        assert o[k] == o_again[k], k
        assert abs(o[k] - w[k]) <= 1e-6 * scale, k
        assert abs(o[k] - o_two[k]) <= 2e-6 * scale, k
    assert np.abs(o["pop"] - w["pop"]).max() <= 1e-6 * scale
