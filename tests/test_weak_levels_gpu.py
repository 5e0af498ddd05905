"""Levels of a site far below its strongest one keep their own digits through the FP64 potential, the 1D steps and the
pull-back: spin mixing grows from seeds many orders of magnitude below the field.

References: the Taylor series of U in numpy's long double, level by level, K by the oracle (it acts on each level
by itself), and the gradient of the step's definition in FP64 torch.  A level's error is measured against what reaches it in the
step: its own size and, in U, what the other levels add.
Tolerances: U 16 roundings of 2^-53 of that; three steps 1e-13 within the 24 sites they reach (four roundings a
step in K, as the other 1D tests); the pull-back 1e-13 of the level's largest component (sums of about a hundred terms).
"""
import numpy as np
import pytest

import oracle
from paper_1907_12834_gb300 import inputs as I
from test_fixed_host import reference

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1907_12834_gb300 import qlga  # noqa: E402
from perf import cases  # noqa: E402

G = (1.0, 0.8, -0.6)
SEEDS = {"polar": (0, 1, 2, 1, 0), "ends": (2, 0, 1, 0, 2), "chain": (4, 3, 2, 1, 0), "even": (2, 2, 2, 2, 2)}


def _state(kind, seed, rng, nx, ny=1, scale=0.04):
    """Level m of size seed^(2 - k) for k = SEEDS[kind][m], one at full size."""
    k = np.array(SEEDS[kind], dtype=float)
    w = seed ** (0.5 * (k.max() - k))
    return I.random_state(rng, nx, ny, scale=scale) * w[:, None, None, None, None]


def _sites(st):  # (5, 1, nx, 2, 2) -> (nx, 5, 2)
    z = st[:, 0, :, :, 0] + 1j * st[:, 0, :, :, 1]
    return np.ascontiguousarray(np.moveaxis(z, 0, 1))


def _reached(x, g):
    """What reaches each level in U: |x_m| + sum_j |V_mj| |x_j| with the moduli's sums in V."""
    p, a = np.abs(x[:, :, 0] + x[:, :, 1]), np.abs(x).sum(axis=2)
    n, c = p ** 2, [1.0, 1.5 ** 0.5, 1.5 ** 0.5, 1.0]
    rho = n.sum(axis=1, keepdims=True)
    fp = 2 * sum(c[i] * p[:, i] * p[:, i + 1] for i in range(4))
    out = a * (1 + (abs(g[0]) + 4 * abs(g[1]) + abs(g[2])) * rho)
    out += abs(g[2]) / 5 * p[:, ::-1] * (p[:, ::-1] * a).sum(axis=1, keepdims=True)
    for m in range(4):
        out[:, m] += abs(g[1]) * c[m] * fp * a[:, m + 1]
        out[:, m + 1] += abs(g[1]) * c[m] * fp * a[:, m]
    return out


@pytest.mark.parametrize("kind", list(SEEDS))
@pytest.mark.parametrize("seed", [1e-3, 1e-10, 1e-40, 1e-180])
@pytest.mark.parametrize("g", [G, (1.0, 0.1, 1.0)])
def test_potential(kind, seed, g):
    nx = 300
    st = _state(kind, seed, np.random.default_rng(7), nx)
    with qlga.Lattice(1, nx, precision=64, g=g) as lat:
        lat.load_state(st)
        lat.apply_potential(1.0)
        got = _sites(lat.get_state())
    x = _sites(st)
    err = np.abs(got - reference(x, g)).max(axis=2).astype(np.float64)
    assert np.all(err <= 16 * 2.0 ** -53 * _reached(x, g)), (err / np.maximum(_reached(x, g), 1e-300)).max(axis=0) * 2.0 ** 53


# ten, five and one lane per site
@pytest.mark.parametrize("L,steps", [(61, 3), (4097, 3), (33001, 1)])
@pytest.mark.parametrize("kind,seed", [("polar", 1e-10), ("ends", 1e-6), ("chain", 1e-12), ("even", 1.0)])
def test_steps_1d(L, steps, kind, seed):
    st = _state(kind, seed, np.random.default_rng(L), L)
    ref, size = st.copy(), np.abs(st).max(axis=(1, 3, 4))
    cfg = oracle.make_cfg(1, L, 1, *G)
    for _ in range(steps):
        x = _sites(ref)
        size = np.maximum(size, _reached(x, G).T)
        z = np.moveaxis(reference(x, G).astype(np.complex128), 1, 0)
        ref[:, 0, :, :, 0], ref[:, 0, :, :, 1] = z.real, z.imag
        oracle.apply_kinetic(ref, cfg)
    with qlga.Lattice(1, L, precision=64, g=G) as lat:
        lat.load_state(st)
        lat.step(steps)
        got = lat.get_state()
    err = np.abs(got - ref).max(axis=(1, 3, 4))
    near = np.max([np.roll(size, k, axis=1) for k in range(-24, 25)], axis=0)
    assert np.all(err <= 1e-13 * near), (err / near).max(axis=1)


@pytest.mark.parametrize("kind,seed", [("polar", 1e-10), ("ends", 1e-6), ("chain", 1e-12), ("even", 1.0)])
@pytest.mark.parametrize("cot_kind", ["even", "polar", "chain"])
@pytest.mark.parametrize("nx,ny", [(70, 1), (37, 12)])
def test_pull_back(kind, seed, cot_kind, nx, ny):
    rng = np.random.default_rng(nx)
    st = torch.tensor(_state(kind, seed, rng, nx, ny), device="cuda")
    cot = torch.tensor(_state(cot_kind, 1e-9, rng, nx, ny, 1.0), device="cuda")
    x, g = st.clone().requires_grad_(True), torch.tensor(G, dtype=torch.float64, device="cuda", requires_grad=True)
    (cases._join(*cases._step(*cases._pair(x if ny > 1 else x.reshape(5, nx, 2, 2)), [g[0], g[1], g[2]], cases._grid_shifts(ny)))
     .reshape(cot.shape) * cot).sum().backward()
    with qlga.Lattice(1 if ny == 1 else 2, nx, ny, precision=64, g=G) as lat:
        got, dg = lat.adjoint_step(st, cot)
    ref = x.grad.reshape(cot.shape)
    for m in range(5):
        assert (got[m] - ref[m]).abs().max() <= 1e-13 * ref[m].abs().max(), m
    assert np.abs(dg - g.grad.cpu().numpy()).max() <= 1e-12 * g.grad.abs().max().item()
