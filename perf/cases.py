"""Performance cases of the spin-2 QLGA framework: what its users run, through its public entry points.

Every case starts from a state on the GPU (solitons in 1D, vortex dipoles in 2D, at the lattice
scaling epsilon = 0.1 of the paper's runs) and takes the whole call: load, steps, read-out.

  run       Lattice: load a state, n steps, observables, the state back (plain or interleaved)
  batch     Batch: many independent lattices of uneven size and couplings, n steps, observables
  gradient  evolve() and the objectives under autograd: gradients of the state and the couplings
  snapshot  Lattice: a stored state is loaded and analysed (observables and the per-site fields)

The 64-bit values (`exact`) come from plain torch: collide and stream as the sweeps of the paper's
operator product, exp(-i delta V) as its Taylor series on V itself.
"""
import ctypes
import math

import torch
from torch.utils.checkpoint import checkpoint

from paper_1907_12834_gb300 import qlga

EPS = 0.1
G_SOLITON = (1.0, -0.5, 0.2)        # the paper's soliton profiles
G_NONINTEGRABLE = (1.0, 0.8, -0.6)  # soliton scattering beyond the profile couplings
G_VORTEX = (1.0, 0.1, 1.0)          # the paper's vortex scattering
WEIGHTS = (1.0, 50.0, 0.02)         # of the m = 0 population, the singlet fraction and the energy in a loss
DEVICE = "cuda" if torch.cuda.is_available() else "cpu"


def listed():
    return [
        # a single stationary soliton, checked for its phase and norm: the smallest lattice, where a
        # step is a few microseconds of latency
        {"name": "run 1d f64 1024", "kind": "run", "precision": 64, "nx": 1024, "ny": 1, "steps": 100,
         "interleave": False, "couplings": "soliton"},
        # two-soliton scattering in FP32 and FP64: 20000 steps in all, read out every hundred
        {"name": "run 1d f32 16384", "kind": "run", "precision": 32, "nx": 16384, "ny": 1, "steps": 100,
         "interleave": False, "couplings": "soliton"},
        {"name": "run 1d f64 16384", "kind": "run", "precision": 64, "nx": 16384, "ny": 1, "steps": 100,
         "interleave": False, "couplings": "nonintegrable"},
        # vortex scattering on a lattice that stays in the L2 cache (the size of the gradient runs)
        {"name": "run 2d f32 512", "kind": "run", "precision": 32, "nx": 512, "ny": 512, "steps": 32,
         "interleave": False, "couplings": "vortex"},
        # vortex scattering at the benchmark's size: the largest call
        {"name": "run 2d f32 4096", "kind": "run", "precision": 32, "nx": 4096, "ny": 4096, "steps": 12,
         "interleave": False, "couplings": "vortex"},
        # the FP64 run that the FP32 one is judged by
        {"name": "run 2d f64 1024", "kind": "run", "precision": 64, "nx": 1024, "ny": 1024, "steps": 10,
         "interleave": False, "couplings": "vortex"},
        # a lattice whose sides fit no tile
        {"name": "run 2d f32 1000x701", "kind": "run", "precision": 32, "nx": 1000, "ny": 701, "steps": 20,
         "interleave": False, "couplings": "vortex"},
        # the interleaved step, U^(1/8) before every kinetic block
        {"name": "run 2d f32 1024 ilv", "kind": "run", "precision": 32, "nx": 1024, "ny": 1024, "steps": 8,
         "interleave": True, "couplings": "vortex"},
        # a scan: 256 scattering runs of uneven length and couplings
        {"name": "batch 1d f32 256", "kind": "batch", "precision": 32, "runs": 256, "lmin": 2048, "lmax": 65536,
         "layout": 1910, "steps": 40},
        # gradients of final populations, singlet fraction and (a little) energy on the vortex lattice
        {"name": "gradient 2d f32 512", "kind": "gradient", "precision": 32, "nx": 512, "ny": 512, "steps": 24,
         "checkpoint_every": 10},
        {"name": "gradient 2d f64 256", "kind": "gradient", "precision": 64, "nx": 256, "ny": 256, "steps": 12,
         "checkpoint_every": 5},
        # a stored snapshot of the benchmark lattice: conserved quantities and the fields to plot
        {"name": "snapshot 2d f32 4096", "kind": "snapshot", "precision": 32, "nx": 4096, "ny": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run1d", "run1d", "run2d", "run2d", "batch", "gradient", "snapshot"])
    prec = rng.choice([32, 64])
    if kind == "run1d":
        nx = _log_int(rng, 256, 262144 if prec == 32 else 65536)
        return {"kind": "run", "precision": prec, "nx": nx, "ny": 1, "steps": rng.randrange(21, 120),
                "interleave": False, "couplings": rng.choice(["soliton", "nonintegrable"])}
    if kind == "run2d":
        hi = 4096 if prec == 32 else 1024
        nx, ny = _log_int(rng, 96, hi), _log_int(rng, 96, hi)
        ilv = rng.random() < 0.2
        if ilv:
            nx, ny = min(nx, 1024), min(ny, 1024)
        if rng.random() < 0.5:  # half of them on the fused kernels' widths
            nx = max(96, nx // 32 * 32)
        cost = nx * ny * (8 if ilv else 1) * (1 if prec == 32 else 20)
        steps = max(2, min(rng.randrange(8, 33), 150_000_000 // cost))
        return {"kind": "run", "precision": prec, "nx": nx, "ny": ny, "steps": steps, "interleave": ilv,
                "couplings": "vortex"}
    if kind == "batch":
        runs = rng.randrange(16, 257)
        return {"kind": "batch", "precision": 32, "runs": runs, "lmin": rng.randrange(1024, 4096),
                "lmax": _log_int(rng, 8192, 65536), "layout": rng.randrange(1 << 20), "steps": rng.randrange(11, 41)}
    if kind == "gradient":
        hi = 512 if prec == 32 else 256
        nx, ny = _log_int(rng, 64, hi), _log_int(rng, 64, hi)
        return {"kind": "gradient", "precision": prec, "nx": nx, "ny": ny, "steps": rng.randrange(5, 25 if prec == 32 else 13),
                "checkpoint_every": rng.randrange(2, 12)}
    nx, ny = _log_int(rng, 256, 4096), _log_int(rng, 256, 4096)
    if prec == 64:
        nx, ny = min(nx, 2048), min(ny, 2048)
    return {"kind": "snapshot", "precision": prec, "nx": nx, "ny": ny}


# ------------------------------------------------------------------ inputs

def _couplings(case):
    return {"soliton": G_SOLITON, "nonintegrable": G_NONINTEGRABLE, "vortex": G_VORTEX}[case.get("couplings", "vortex")]


def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed) * 7919 + 13)


def _uniform(gen, lo, hi, n=1):
    return (lo + (hi - lo) * torch.rand(n, generator=gen, device=DEVICE, dtype=torch.float64)).tolist()


def _spin_levels(theta, phi):
    """The five levels of a spin-coherent state turned by theta about y and phi about z."""
    c, s = math.cos(theta / 2), math.sin(theta / 2)
    w = [c ** 4, 2 * c ** 3 * s, math.sqrt(6) * c * c * s * s, 2 * c * s ** 3, s ** 4]
    return [complex(w[i] * math.cos((2 - i) * phi), -w[i] * math.sin((2 - i) * phi)) for i in range(5)]


def _solitons(L, gen):
    """Two bright solitons sqrt(2) sech in turned spin states, opposite kicks, a relative phase."""
    j = torch.arange(L, device=DEVICE, dtype=torch.float64)
    kappa, rel, t1, t2, p1, p2 = _uniform(gen, 0.0, 1.0, 6)
    p = 2 * math.pi * round((0.05 + 0.25 * kappa) * L / (2 * math.pi)) / L
    psi = torch.zeros(5, L, device=DEVICE, dtype=torch.complex128)
    for at, theta, phi, kick, phase in ((0.25, t1, p1, p, 0.0), (0.75, t2, p2, -p, rel)):
        prof = math.sqrt(2.0) / torch.cosh((EPS * (j - at * L)).clamp(-300, 300))
        wave = prof * torch.exp(1j * (kick * j + 2 * math.pi * phase))
        for m, w in enumerate(_spin_levels(math.pi * theta, 2 * math.pi * phi)):
            psi[m] += w * wave
    return psi


def _vortices(nx, ny, gen):
    """A vortex dipole in m = +2 and its counter-rotating partner in m = -2, unit background, and
    the other levels at a tenth of it."""
    x = torch.arange(nx, device=DEVICE, dtype=torch.float64)[None, :]
    y = torch.arange(ny, device=DEVICE, dtype=torch.float64)[:, None]
    sep = nx / 4 if nx < 256 else 64.0
    psi = torch.empty(5, ny, nx, device=DEVICE, dtype=torch.complex128)
    for m in range(5):
        kx, ky, ph = _uniform(gen, -3.0, 3.0, 3)
        wave = 2 * math.pi * (round(kx) * x / nx + round(ky) * y / ny) + ph
        amp = torch.full((ny, nx), 0.1, device=DEVICE, dtype=torch.float64)
        if m in (0, 4):
            amp = torch.ones((ny, nx), device=DEVICE, dtype=torch.float64)
            for sign in (-1, 1):
                dx, dy = x - (nx / 2 + 0.5 + sign * sep / 2), y - (ny / 2 + 0.5)
                r2 = EPS * EPS * (dx * dx + dy * dy)
                amp = amp * torch.sqrt((0.1 * r2 * r2 + 0.3 * r2) / (0.1 * r2 * r2 + 0.6 * r2 + 1))
                wave = wave + (sign if m == 0 else -sign) * torch.atan2(dy, dx)
        psi[m] = torch.polar(amp, wave)
    return psi


def _state(psi, gen, mix, dtype):
    """The framework's state (5, ny, nx, 2, 2) of a physical field: a = b = eps psi / 2, and for a
    run that has settled (mix > 0) a difference a - b of mix times the field."""
    z = torch.view_as_real(0.5 * EPS * psi)  # (5, ..., 2)
    ny, nx = (1, psi.shape[1]) if psi.dim() == 2 else psi.shape[1:]
    z = z.reshape(5, ny, nx, 1, 2).expand(5, ny, nx, 2, 2).to(dtype, copy=True)
    if mix:
        d = torch.randn(5, ny, nx, 2, generator=gen, device=DEVICE, dtype=torch.float32)
        scale = (0.5 * EPS * mix) * psi.abs().reshape(5, ny, nx, 1).to(torch.float32)
        d = d * scale
        z[..., 0, :] += d
        z[..., 1, :] -= d
    return z.contiguous()


def _inputs(case, seed):
    gen = _generator(seed)
    dtype = torch.float32 if case["precision"] == 32 else torch.float64
    if case["kind"] == "batch":
        lengths, G = [], []  # the lengths go with the case, the couplings and states with the seed
        for u in _uniform(_generator(case["layout"]), 0.0, 1.0, case["runs"]):
            lengths.append(int(round(case["lmin"] * (case["lmax"] / case["lmin"]) ** u)))
        for _ in lengths:
            G.append([1.0] + _uniform(gen, -1.0, 1.0, 2))
        return lengths, G, [_state(_solitons(L, gen), gen, 0.0, dtype).reshape(-1) for L in lengths]
    if case["ny"] == 1:
        return _state(_solitons(case["nx"], gen), gen, 0.0, dtype)
    # a vortex lattice spends its run with |a - b| near |a + b|; gradients start from a fresh state
    return _state(_vortices(case["nx"], case["ny"], gen), gen, 0.0 if case["kind"] == "gradient" else 0.5, dtype)


# ------------------------------------------------------------------ the framework's calls

_OBS = ("norm_qubit", "norm_boson", "magnetisation", "energy", "singlet_re", "singlet_im", "singlet_fraction")


def _obs_row(o):
    return [o[k] for k in _OBS] + o["pop"].tolist()


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        lengths, G, parts = x
        batch = qlga.Batch(lengths, G, precision=case["precision"], epsilon=EPS)
        flat = torch.cat(parts)
        return {"case": case, "batch": batch, "x": flat, "out": torch.empty_like(flat)}
    if kind == "gradient":
        g = torch.tensor(G_VORTEX, dtype=x.dtype, device=DEVICE)
        w = torch.tensor(WEIGHTS, dtype=torch.float64, device=DEVICE)
        return {"case": case, "x": x, "g": g, "w": w}
    lat = qlga.Lattice(1 if case["ny"] == 1 else 2, case["nx"], case["ny"], precision=case["precision"],
                       g=_couplings(case), epsilon=EPS, interleave=int(case.get("interleave", False)))
    out = {"case": case, "lat": lat, "x": x}
    if kind == "snapshot":
        out["fields"] = torch.empty((11, case["ny"], case["nx"]), dtype=x.dtype, device=DEVICE)
    else:
        out["out"] = torch.empty_like(x)
    return out


def run(state):
    case, x = state["case"], state["x"]
    kind = case["kind"]
    if kind == "run":
        lat = state["lat"]
        lat.load_state(x)
        lat.step(case["steps"])
        obs = lat.observables()
        return {"state": lat.get_state(state["out"]), "obs": torch.tensor(_obs_row(obs), dtype=x.dtype)}
    if kind == "snapshot":
        lat = state["lat"]
        lat.load_state(x)
        obs = lat.observables()
        qlga.qlga_fields(lat.handle, state["fields"].data_ptr(), qlga.QLGA_DEVICE)
        return {"fields": state["fields"], "obs": torch.tensor(_obs_row(obs), dtype=x.dtype)}
    if kind == "batch":
        batch, lib = state["batch"], qlga.load_library()
        h = ctypes.c_void_p(batch.handle)
        qlga._check(lib.qlga_batch_load_state(h, ctypes.c_void_p(x.data_ptr()), qlga.QLGA_DEVICE), "load")
        batch.step(case["steps"])
        obs = batch.observables()
        qlga._check(lib.qlga_batch_get_state(h, ctypes.c_void_p(state["out"].data_ptr()), qlga.QLGA_DEVICE), "get")
        return {"state": state["out"], "obs": torch.tensor([_obs_row(o) for o in obs], dtype=x.dtype)}
    x0 = x.detach().requires_grad_(True)
    g = state["g"].detach().requires_grad_(True)
    xn = qlga.evolve(x0, g, case["steps"], case["checkpoint_every"])
    values = qlga.objectives(xn, g)
    loss = (values * state["w"]).sum()
    loss.backward()
    return {"values": values.detach().to(x.dtype), "dx": x0.grad, "dg": g.grad}


# ------------------------------------------------------------------ work

def work(case):
    # operations of a site and step: the integer stencil of an axis (24 taps on 5 complex levels),
    # the second axis as eight collides, the quadratic forms and phases of U, and its Taylor terms
    # (two vectors, 66 multiply-adds each) to the degree that the tolerance of the type asks for
    reals = 4 if case["precision"] == 32 else 8
    if case["kind"] == "batch":
        ratio = case["lmax"] / case["lmin"]
        sites = int(case["runs"] * (case["lmax"] - case["lmin"]) / math.log(ratio))
        two_d, steps = False, case["steps"]
    else:
        sites, two_d, steps = case["nx"] * case["ny"], case["ny"] > 1, case.get("steps", 0)
    state = 20 * reals * sites
    if case["kind"] == "snapshot":
        return {"bytes": state + 11 * reals * sites, "flops": 250 * sites}
    degree = 2 if case["precision"] == 32 else 5
    u = 250 + 264 * degree
    per_step = 240 + (160 if two_d else 0) + u
    if case.get("interleave"):
        per_step = (8 if two_d else 4) * u + (320 if two_d else 160)
    if case["kind"] == "gradient":
        # forward, the recomputed segment, the adjoint stencil and seven times the Taylor work
        per_step = 2 * per_step + 240 + 160 + 400 + 7 * 264 * degree
        return {"bytes": 4 * state, "flops": per_step * sites * steps}
    # one read and one write of the state a step where it is larger than the L2 cache, else in all
    passes = steps if state > 100e6 else 1
    return {"bytes": 2 * state * passes, "flops": per_step * sites * steps}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch

def _v_apply(p, x, g):
    """V(p) x of the spin-2 interaction: density, spin density and singlet pair."""
    g0, g1, g2 = g
    n = [p[i].real ** 2 + p[i].imag ** 2 for i in range(5)]
    rho = n[0] + n[1] + n[2] + n[3] + n[4]
    fz = 2 * (n[0] - n[4]) + n[1] - n[3]
    r = math.sqrt(1.5)
    fp = 2 * (p[0].conj() * p[1] + p[3].conj() * p[4] + r * (p[1].conj() * p[2] + p[2].conj() * p[3]))
    s = [p[4].conj(), -p[3].conj(), p[2].conj(), -p[1].conj(), p[0].conj()]
    t = sum(s[i].conj() * x[i] for i in range(5)) * (g2 / 5)
    c = [1.0, r, r, 1.0]
    y = [(g0 * rho + (2 - i) * g1 * fz) * x[i] + s[i] * t for i in range(5)]
    for i in range(4):
        y[i] = y[i] + g1 * c[i] * fp.conj() * x[i + 1]
        y[i + 1] = y[i + 1] + g1 * c[i] * fp * x[i]
    return y


def _terms(p, g, delta):
    """Taylor terms of exp(-i delta V) that reach below 1e-19 at the densest site."""
    rho = float(sum(z.real ** 2 + z.imag ** 2 for z in p).max())
    bound = abs(delta) * rho * max(float((abs(g[0]) + 4 * abs(g[1]) + abs(g[2])).max())
                                   if isinstance(g[0], torch.Tensor) else abs(g[0]) + 4 * abs(g[1]) + abs(g[2]), 1e-30)
    n, term = 1, bound
    while term > 1e-19 and n < 60:
        n += 1
        term *= bound / n
    return n


def _potential(a, b, g, delta):
    p = [a[i] + b[i] for i in range(5)]
    with torch.no_grad():
        n = _terms([z.detach() for z in p], [v.detach() if isinstance(v, torch.Tensor) else v for v in g], delta)
    out = []
    for x in (a, b):
        v = x
        for k in range(n, 0, -1):
            w = _v_apply(p, v, g)
            v = [x[i] - (1j * delta / k) * w[i] for i in range(5)]
        out.append(v)
    return out


def _collide(a, b):
    s, d = 0.5 * (1 - 1j), 0.5 * (1 + 1j)
    return [s * x + d * y for x, y in zip(a, b)], [d * x + s * y for x, y in zip(a, b)]


def _block(a, b, qubit, shift):
    """I'_c = S_c C S_c^T C of one axis: shift(z, +1) moves a field one site toward +x."""
    a, b = _collide(a, b)
    if qubit == 2:
        b = [shift(z, -1) for z in b]
    else:
        a = [shift(z, -1) for z in a]
    a, b = _collide(a, b)
    if qubit == 2:
        b = [shift(z, 1) for z in b]
    else:
        a = [shift(z, 1) for z in a]
    return a, b


def _step(a, b, g, shifts, interleave=False):
    if not interleave:
        a, b = _potential(a, b, g, 1.0)
    for shift in shifts:
        for qubit in (2, 2, 1, 1):
            if interleave:
                a, b = _potential(a, b, g, 1.0 / (4 * len(shifts)))
            a, b = _block(a, b, qubit, shift)
    return a, b


def _pair(x):
    """The five levels of both qubits of a state tensor (5, ny, nx, 2, 2), in 64 bits."""
    z = torch.view_as_complex(x.double().contiguous())
    return [z[m, ..., 0] for m in range(5)], [z[m, ..., 1] for m in range(5)]


def _join(a, b):
    return torch.stack([torch.stack([torch.view_as_real(a[m]), torch.view_as_real(b[m])], dim=-2) for m in range(5)])


def _grid_shifts(ny):
    shifts = [lambda z, k: torch.roll(z, k, dims=-1)]
    if ny > 1:
        shifts.append(lambda z, k: torch.roll(z, k, dims=-2))
    return shifts


def _densities(p, g):
    """rho, |F|^2, F_z, F_+, theta = psi^T J psi of a boson field."""
    n = [z.real ** 2 + z.imag ** 2 for z in p]
    rho = n[0] + n[1] + n[2] + n[3] + n[4]
    fz = 2 * (n[0] - n[4]) + n[1] - n[3]
    r = math.sqrt(1.5)
    fp = 2 * (p[0].conj() * p[1] + p[3].conj() * p[4] + r * (p[1].conj() * p[2] + p[2].conj() * p[3]))
    theta = 2 * p[0] * p[4] - 2 * p[1] * p[3] + p[2] * p[2]
    return rho, fz ** 2 + fp.real ** 2 + fp.imag ** 2, fz, fp, theta


def _sums(a, b, g, shifts):
    """Per-site terms of the observables: qubit norm, boson norm, energy, singlet, theta^2, rho^2, populations."""
    pop = [a[m].real ** 2 + a[m].imag ** 2 + b[m].real ** 2 + b[m].imag ** 2 for m in range(5)]
    p = [a[m] + b[m] for m in range(5)]
    rho, f2, _, _, theta = _densities(p, g)
    t2 = theta.real ** 2 + theta.imag ** 2
    e = 0.5 * g[0] * rho ** 2 + 0.5 * g[1] * f2 + 0.1 * g[2] * t2
    for shift in shifts:
        for z in p:
            d = shift(z, -1) - z
            e = e + d.real ** 2 + d.imag ** 2
    return [sum(pop), rho, e, theta.real, theta.imag, t2, rho ** 2] + pop


def _obs_of(s):
    nq, nb, e, tr, ti, t2, r2 = s[:7]
    pop = s[7:]
    mag = sum((2 - m) * pop[m] for m in range(5))
    return [nq, nb, mag, e, tr / math.sqrt(5), ti / math.sqrt(5), t2 / r2] + pop


def _fields(p):
    rho, _, fz, fp, theta = _densities(p, None)
    fperp, a00 = fp.abs(), theta.abs() / math.sqrt(5)
    nrm = torch.sqrt(fz ** 2 + fperp ** 2 + a00 ** 2)
    safe = torch.where(nrm > 0, nrm, torch.ones_like(nrm))
    out = [fz, fperp, a00, fz.abs() / safe, fperp / safe, a00 / safe]

    def wrap(d):
        return d - 2 * math.pi * torch.round(d / (2 * math.pi))

    for z in p:
        ph = torch.angle(z)
        vx = wrap(torch.roll(ph, -1, -1) - torch.roll(ph, 1, -1)) / 2
        vy = wrap(torch.roll(ph, -1, -2) - torch.roll(ph, 1, -2)) / 2
        out.append((torch.roll(vy, -1, -1) - torch.roll(vy, 1, -1) - torch.roll(vx, -1, -2) + torch.roll(vx, 1, -2)) / 2)
    return torch.stack(out)


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        with torch.no_grad():
            return _exact_batch(case, *x)
    shifts = _grid_shifts(case["ny"])
    if kind == "gradient":
        return _exact_gradient(case, x, shifts)
    with torch.no_grad():
        a, b = _pair(x)
        g = _couplings(case)
        if kind == "snapshot":
            obs = torch.stack(_obs_of([t.sum() for t in _sums(a, b, g, shifts)]))
            return {"fields": _fields([a[m] + b[m] for m in range(5)]), "obs": obs}
        del x
        for _ in range(case["steps"]):
            a, b = _step(a, b, g, shifts, case["interleave"])
        obs = torch.stack(_obs_of([t.sum() for t in _sums(a, b, g, shifts)]))
        return {"state": _join(a, b), "obs": obs}


def _exact_batch(case, lengths, G, parts):
    """The runs end to end as one field; a shift reads each run's own neighbour."""
    L = torch.tensor(lengths, device=DEVICE)
    run = torch.repeat_interleave(torch.arange(len(lengths), device=DEVICE), L)
    start = (torch.cumsum(L, 0) - L)[run]
    j = torch.arange(len(run), device=DEVICE) - start
    at = {k: start + (j - k) % L[run] for k in (-1, 1)}  # shift +1: c(j) <- c(j - 1)
    a, b = [], []
    for m in range(5):
        z = [torch.view_as_complex(s.view(5, -1, 2, 2)[m].double().contiguous()) for s in parts]
        a.append(torch.cat([t[:, 0] for t in z]))
        b.append(torch.cat([t[:, 1] for t in z]))
    g = [torch.tensor([r[k] for r in G], dtype=torch.float64, device=DEVICE)[run] for k in range(3)]
    shifts = [lambda z, k: z[at[k]]]
    for _ in range(case["steps"]):
        a, b = _step(a, b, g, shifts)
    zero = torch.zeros(len(lengths), dtype=torch.float64, device=DEVICE)
    obs = torch.stack(_obs_of([zero.index_add(0, run, t) for t in _sums(a, b, g, shifts)]), dim=1)
    whole = _join(a, b)
    pieces = [t.reshape(-1) for t in torch.split(whole, lengths, dim=1)]
    return {"state": torch.cat(pieces), "obs": obs}


def _exact_gradient(case, x, shifts):
    x0 = x.double().requires_grad_(True)
    gt = torch.tensor(G_VORTEX, dtype=torch.float64, device=DEVICE, requires_grad=True)

    def one(s, gt):
        return _join(*_step(*_pair(s), [gt[0], gt[1], gt[2]], shifts))

    s = x0
    for _ in range(case["steps"]):
        s = checkpoint(one, s, gt, use_reentrant=False)
    a, b = _pair(s)
    g = [gt[0], gt[1], gt[2]]
    sums = [t.sum() for t in _sums(a, b, g, shifts)]
    values = torch.stack([sums[7 + 2], sums[5] / sums[6], sums[2]])
    (values * torch.tensor(WEIGHTS, dtype=torch.float64, device=DEVICE)).sum().backward()
    return {"values": values.detach(), "dx": x0.grad, "dg": gt.grad}
