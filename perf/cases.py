"""Workloads of the solver, from one residual evaluation to a whole 512^3 solve, each
through the public entry points of ``paper_1303_0008_gb300.mg``.

  listed()             the named cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  inputs on the GPU and the handle that a program keeps
  run(state)           one pass; returns its outputs
  work(case)           bytes and operations that one pass cannot do without
  exact(case, seed)    the outputs in plain torch, float64

Density contrasts are lognormal fields (P(k) ~ k^-2), the stand-ins for N-body
densities that the repository's other workloads use; the screening strength is given
by the Vainshtein radius r_v in cells of a reference top-hat, and sign = -1 flips alpha
and kappa together (the self-accelerating branch).
"""
from __future__ import annotations

import math

import torch

from paper_1303_0008_gb300 import inputs, mg

TOL = 1e-8
DEV = "cuda"


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # The residual and its norms of a small grid, as a driver checks a field that it
        # holds: a call of some tens of microseconds.
        {"name": "residual_64", "kind": "residual", "n": 64, "r_v": 8.0, "sigma": 1.5, "sign": 1,
         "rhs": False},
        # Two smoothing sweeps with a right-hand side: a user's own cycle around the
        # library's smoother.
        {"name": "smooth_256", "kind": "smooth", "n": 256, "r_v": 8.0, "sigma": 1.5, "sign": 1,
         "rhs": True, "sweeps": 2},
        # Both grid transfers at a ragged side.
        {"name": "transfer_300", "kind": "transfer", "n": 300},
        # Density of one simulation step: 256^3 particles onto 256^3 cells (TSC).
        {"name": "deposit_256", "kind": "deposit", "n": 256, "side": 256, "scheme": 2,
         "equal_mass": True},
        # Small box: bound by latency and launches.
        {"name": "fp64_32", "kind": "solve", "n": 32, "r_v": 8.0, "sigma": 1.5, "sign": 1,
         "mixed": False, "nu_pre": 2, "nu_post": 2, "inner": 3},
        # The everyday solve with the default options.
        {"name": "fp64_128", "kind": "solve", "n": 128, "r_v": 8.0, "sigma": 1.5, "sign": 1,
         "mixed": False, "nu_pre": 2, "nu_post": 2, "inner": 3},
        # alpha = 0: the Poisson equation (Newtonian potential, or no screening).
        {"name": "poisson_256", "kind": "solve", "n": 256, "r_v": 0.0, "sigma": 1.5, "sign": 1,
         "mixed": False, "nu_pre": 2, "nu_post": 2, "inner": 3},
        # The benchmark's box in FP64, more sweeps per cycle as tuning chooses them there.
        {"name": "fp64_512", "kind": "solve", "n": 512, "r_v": 8.0, "sigma": 1.5, "sign": 1,
         "mixed": False, "nu_pre": 4, "nu_post": 4, "inner": 3},
        # Mixed precision at a side that is no power of two, self-accelerating branch.
        {"name": "mixed_192", "kind": "solve", "n": 192, "r_v": 4.0, "sigma": 1.5, "sign": -1,
         "mixed": True, "nu_pre": 2, "nu_post": 2, "inner": 3},
        # The benchmark's box in mixed precision with its tuned sweep counts.
        {"name": "mixed_512", "kind": "solve", "n": 512, "r_v": 16.0, "sigma": 2.0, "sign": 1,
         "mixed": True, "nu_pre": 5, "nu_post": 4, "inner": 4},
        # Many independent boxes of several sizes at once (parameter scans).
        {"name": "batch_64", "kind": "batch", "count": 64, "largest": 128, "mixed": True},
        # A domain with two refinement levels over its dense regions (a sixteenth of the
        # volume, and 512 patches inside it).
        {"name": "refined_256", "kind": "refined", "n": 256, "r_v": 8.0, "sigma": 1.5, "sign": 1,
         "patches": 16384},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(rng, lo, hi):
    """An even side, spread over the logarithm: odd multiples of 2 among them."""
    return 2 * max(lo // 2, min(hi // 2, round(_log_uniform(rng, lo, hi) / 2)))


#: sides whose hierarchy ends at 4, 6, 10 or 14 cells
_SIDES = (24, 28, 32, 40, 48, 56, 64, 80, 96, 112, 128, 160, 192, 224, 256, 320, 384, 448)


def _side(rng, lo, hi):
    x = _log_uniform(rng, lo, hi)
    return min((s for s in _SIDES if lo <= s <= hi), key=lambda s: abs(math.log(s / x)))


def draw(rng):
    kind = rng.choice(["residual", "smooth", "transfer", "deposit", "solve", "solve", "solve",
                       "solve", "batch", "refined"])
    phys = {"r_v": round(_log_uniform(rng, 2.0, 16.0), 3), "sigma": round(rng.uniform(0.5, 2.0), 3),
            "sign": rng.choice([1, -1])}
    if kind == "residual":
        return {"kind": kind, "n": _even(rng, 16, 256), **phys, "rhs": rng.random() < 0.5}
    if kind == "smooth":
        return {"kind": kind, "n": _even(rng, 16, 384), **phys, "rhs": rng.random() < 0.5,
                "sweeps": rng.randint(1, 4)}
    if kind == "transfer":
        return {"kind": kind, "n": _even(rng, 16, 512)}
    if kind == "deposit":
        return {"kind": kind, "n": _side(rng, 24, 384), "side": rng.randint(24, 320),
                "scheme": rng.choice([1, 2]), "equal_mass": rng.random() < 0.5}
    if kind == "solve":
        mixed = rng.random() < 0.5
        nu = rng.choice([(2, 2), (2, 2), (3, 3), (4, 4), (3, 2)])
        if rng.random() < 0.15:
            phys["r_v"] = 0.0
        return {"kind": kind, "n": _side(rng, 24, 448 if mixed else 320), **phys, "mixed": mixed,
                "nu_pre": nu[0], "nu_post": nu[1], "inner": rng.choice([3, 4])}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(4, 64), "largest": rng.choice([32, 64, 96, 128]),
                "mixed": rng.random() < 0.7}
    n = _side(rng, 64, 256)
    return {"kind": kind, "n": n, "r_v": round(_log_uniform(rng, 2.0, 8.0), 3),
            "sigma": round(rng.uniform(1.0, 1.5), 3), "sign": phys["sign"],
            "patches": round((n // 4) ** 3 * _log_uniform(rng, 0.02, 0.1))}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _parameters(case):
    if case["r_v"] == 0.0:
        return 0.0, float(case["sign"])
    return case["sign"] * inputs.alpha_kappa_for_rv(case["r_v"]), float(case["sign"])


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _poisson(rhs):
    """phi with mean 0 and seven-point Laplacian rhs - mean(rhs) on the periodic unit box."""
    n = rhs.shape[0]
    k = torch.arange(n, dtype=torch.float64, device=rhs.device)
    c = (2.0 * torch.cos(2.0 * math.pi * k / n) - 2.0) * float(n * n)
    ev = c[:, None, None] + c[None, :, None] + c[None, None, :n // 2 + 1]
    ev[0, 0, 0] = 1.0
    f = torch.fft.rfftn(rhs)
    f /= ev
    f[0, 0, 0] = 0.0
    return torch.fft.irfftn(f, s=rhs.shape)


def _field_inputs(case, seed):
    """A density, a field near the solution of its equation with an error at the scale of
    the cells, and a right-hand side: what a cycle holds half-way."""
    n = case["n"]
    alpha, kappa = _parameters(case)
    delta = inputs.lognormal_delta_device(n, case["sigma"], seed)
    phi = _poisson(torch.log1p(delta) * kappa)
    gen = _generator(seed + 1)
    noise = torch.randn((n, n, n), generator=gen, dtype=torch.float64, device=DEV)
    phi += noise * (0.02 / (n * n))
    rhs = None
    if case["rhs"]:
        rhs = 0.05 * torch.randn((n, n, n), generator=gen, dtype=torch.float64, device=DEV)
    return delta, phi.contiguous(), rhs, alpha, kappa


def _particles(case, seed):
    """(3, side^3) positions: a lattice moved by the gradient of a Gaussian potential (the
    Zel'dovich approximation), in lattice order."""
    s = case["side"]
    g = torch.randn((s, s, s), generator=_generator(seed), dtype=torch.float64, device=DEV)
    f = torch.fft.rfftn(g)
    k1 = torch.fft.fftfreq(s, device=DEV, dtype=torch.float64) * s
    kr = torch.fft.rfftfreq(s, device=DEV, dtype=torch.float64) * s
    ks = (kr[None, None, :], k1[None, :, None], k1[:, None, None])  # x, y, z
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    f *= k2 ** -1.5
    f[0, 0, 0] = 0.0
    lattice = (torch.arange(s, device=DEV, dtype=torch.float64) + 0.5) / s
    shape = ((1, 1, s), (1, s, 1), (s, 1, 1))
    pos = torch.empty((3, s, s, s), dtype=torch.float64, device=DEV)
    for a in range(3):
        psi = torch.fft.irfftn(1j * ks[a] * f, s=(s, s, s))
        pos[a] = torch.remainder(lattice.reshape(shape[a]) + psi * (0.015 / psi.std()), 1.0)
    pos = pos.reshape(3, -1).contiguous()
    mass = None
    if not case["equal_mass"]:
        mass = torch.rand(pos.shape[1], generator=_generator(seed + 1), dtype=torch.float64,
                          device=DEV) + 0.5
        mass /= mass.sum()
    return pos, mass


def _batch_specs(case, seed):
    """Sizes, spectra and couplings of the solves: sigma in [0.5, 2.5], r_v in [2, 16]."""
    gen = torch.Generator().manual_seed(seed)
    sizes = [n for n in (32, 64, 96, 128) if n <= case["largest"]]
    out = []
    for k in range(case["count"]):
        u = torch.rand(3, generator=gen, dtype=torch.float64).tolist()
        sign = 1.0 if u[2] < 0.5 else -1.0
        r_v = math.exp(math.log(2.0) + u[1] * math.log(8.0))
        out.append({"n": sizes[k % len(sizes)], "sigma": 0.5 + 2.0 * u[0], "kappa": sign,
                    "alpha": sign * inputs.alpha_kappa_for_rv(r_v)})
    return out


def _patch_values(parent_block, gen):
    """8^3 fine values of each (6^3) parent block, trilinear and cell-centred, times
    1 + 0.1 u: the smallest scales that a refinement resolves."""
    x = parent_block
    for axis in (1, 2, 3):
        lo, mid, hi = (x.narrow(axis, o, 4) for o in (0, 1, 2))
        x = torch.stack((0.25 * lo + 0.75 * mid, 0.75 * mid + 0.25 * hi), dim=axis + 1)
        x = x.flatten(axis, axis + 1)
    u = torch.rand(x.shape, generator=gen, dtype=torch.float64, device=DEV)
    return x * (1.0 + 0.1 * (2.0 * u - 1.0))


def _block_index(origins, n):
    """Index tensors (z, y, x) of the 6^3 cells around the 4^3 blocks at `origins`."""
    o = torch.arange(-1, 5, device=DEV)
    x, y, z = ((origins[:, a, None] + o) % n for a in range(3))
    return z[:, :, None, None], y[:, None, :, None], x[:, None, None, :]


# ---------------------------------------------------------------------------
# State
# ---------------------------------------------------------------------------
class _Handle:
    """A solver handle on torch's current stream, released with its state."""

    def __init__(self, handle):
        self.h = handle
        mg.mg_set_stream(handle, torch.cuda.current_stream())

    def __del__(self):
        mg.mg_destroy_grid(self.h)


def _solver_options(case):
    return mg.options(prec=mg.MG_MIXED if case["mixed"] else mg.MG_FP64, nu_pre=case["nu_pre"],
                      nu_post=case["nu_post"], inner_cycles=case["inner"])


def _refined_levels(case, delta, gen):
    """Origins and density contrast of the two refinement levels: level 2 over the densest
    cells, level 1 over the densest 4^3 blocks of the domain and around level 2."""
    n, count = case["n"], case["patches"]
    nb = n // 4  # blocks of the domain, and patches of level 1, per side
    blocks = delta.reshape(nb, 4, nb, 4, nb, 4).permute(0, 2, 4, 1, 3, 5).reshape(-1, 64)
    peak, cell = blocks.max(dim=1)
    top = peak.topk(count // 32).indices.sort().values
    b2 = torch.stack((top % nb, top // nb % nb, top // (nb * nb)), dim=1)
    cell = cell[top]
    corner = torch.stack((cell % 4, cell // 4 % 4, cell // 16), dim=1) // 2
    # a level-2 patch and the cells around it lie in the 8 level-1 patches at its corner
    for m in range(8):
        x, y, z = ((b2[:, a] + (m >> a & 1) * (2 * corner[:, a] - 1)) % nb for a in range(3))
        peak[(z * nb + y) * nb + x] = math.inf
    first = peak.topk(count).indices.sort().values
    b1 = torch.stack((first % nb, first // nb % nb, first // (nb * nb)), dim=1)
    rho1 = _patch_values((delta + 1.0)[_block_index(4 * b1, n)], gen)
    table = torch.full((nb, nb, nb), -1, dtype=torch.long, device=DEV)
    table[b1[:, 2], b1[:, 1], b1[:, 0]] = torch.arange(count, device=DEV)
    org2 = 2 * (8 * b2 + 4 * corner)
    z, y, x = _block_index(org2 // 2, 2 * n)
    rho2 = _patch_values(rho1[table[z // 8, y // 8, x // 8], z % 8, y % 8, x % 8], gen)
    return [(8 * b1, (rho1 - 1.0).contiguous()), (org2, (rho2 - 1.0).contiguous())]


def _prepare_refined(case, seed):
    alpha, kappa = _parameters(case)
    delta = inputs.lognormal_delta_device(case["n"], case["sigma"], seed)
    levels = _refined_levels(case, delta, _generator(seed + 1))
    grid = _Handle(mg.mg_create_grid(case["n"]))
    for level, (org, _) in enumerate(levels, start=1):
        mg.mg_add_patches(grid.h, level, org.cpu().numpy())
    return {"case": case, "grid": grid, "delta": delta, "zero": torch.zeros_like(delta),
            "levels": [d for _, d in levels], "alpha": alpha, "kappa": kappa}


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("residual", "smooth"):
        delta, phi, rhs, alpha, kappa = _field_inputs(case, seed)
        return {"case": case, "delta": delta, "phi": phi, "rhs": rhs, "alpha": alpha,
                "kappa": kappa, "out": torch.empty_like(phi)}
    if kind == "transfer":
        n, gen = case["n"], _generator(seed)
        fine = torch.randn((n, n, n), generator=gen, dtype=torch.float64, device=DEV)
        coarse = torch.randn((2, n // 2, n // 2, n // 2), generator=gen, dtype=torch.float64,
                             device=DEV)
        return {"case": case, "fine": fine, "coarse": coarse[0], "coarse_ref": coarse[1],
                "restricted": torch.empty_like(coarse[0]), "corrected": torch.empty_like(fine)}
    if kind == "deposit":
        pos, mass = _particles(case, seed)
        n = case["n"]
        return {"case": case, "grid": _Handle(mg.mg_create_grid(n)), "pos": pos, "mass": mass,
                "out": torch.empty((n, n, n), dtype=torch.float64, device=DEV)}
    if kind == "solve":
        alpha, kappa = _parameters(case)
        delta = inputs.lognormal_delta_device(case["n"], case["sigma"], seed)
        grid = _Handle(mg.mg_create_grid(case["n"], _solver_options(case)))
        return {"case": case, "grid": grid, "delta": delta, "zero": torch.zeros_like(delta),
                "alpha": alpha, "kappa": kappa}
    if kind == "batch":
        specs = _batch_specs(case, seed)
        deltas = [inputs.lognormal_delta_device(s["n"], s["sigma"], seed + k)
                  for k, s in enumerate(specs)]
        grid = _Handle(mg.mg_create_batch(
            [s["n"] for s in specs], mg.options(prec=mg.MG_MIXED if case["mixed"] else mg.MG_FP64)))
        return {"case": case, "grid": grid, "specs": specs, "deltas": deltas,
                "zeros": [torch.zeros_like(d) for d in deltas]}
    return _prepare_refined(case, seed)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _field_and_force(h, level, like):
    phi = mg.mg_get_field(h, level, -1, torch.empty_like(like))
    force = mg.mg_get_force(h, level, -1, like.new_empty((3,) + tuple(like.shape)))
    return [phi, force]


def run(state):
    case = state["case"]
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "residual":
        norms = mg.mg_op_residual_noalloc(case["n"], state["phi"], state["delta"], state["rhs"], 0,
                                          state["alpha"], state["kappa"], state["out"],
                                          stream=stream)
        return [state["out"], norms["max"], norms["min"], norms["guards"], norms["nonfinite"]]
    if kind == "smooth":
        out = state["out"].copy_(state["phi"])
        mg.mg_op_smooth(case["n"], out, state["delta"], state["rhs"], 0, state["alpha"],
                        state["kappa"], 0.01, case["sweeps"], stream=stream)
        return out
    if kind == "transfer":
        mg.mg_op_restrict(case["n"], state["fine"], state["restricted"], stream=stream)
        corrected = state["corrected"].copy_(state["fine"])
        mg.mg_op_prolong_correct(case["n"], state["coarse"], state["coarse_ref"], corrected,
                                 stream=stream)
        return [state["restricted"], corrected]
    h = state["grid"].h
    if kind == "deposit":
        mg.mg_assign_density(h, 0, state["pos"], state["mass"], scheme=case["scheme"])
        return mg.mg_get_density(h, 0, -1, state["out"])
    if kind == "solve":
        mg.mg_set_density(h, 0, -1, state["delta"])
        mg.mg_set_field(h, 0, -1, state["zero"])
        mg.mg_solve(h, 0, state["alpha"], state["kappa"], TOL)
        return _field_and_force(h, 0, state["delta"])
    if kind == "batch":
        for k, (delta, zero) in enumerate(zip(state["deltas"], state["zeros"])):
            mg.mg_set_density(h, 0, k, delta)
            mg.mg_set_field(h, 0, k, zero)
        specs = state["specs"]
        mg.mg_solve_batch(h, [0] * len(specs), [s["alpha"] for s in specs],
                          [s["kappa"] for s in specs], TOL)
        return [mg.mg_get_field(h, 0, k, torch.empty_like(d))
                for k, d in enumerate(state["deltas"])]
    mg.mg_set_density(h, 0, -1, state["delta"])
    mg.mg_set_field(h, 0, -1, state["zero"])
    for level, delta in enumerate(state["levels"], start=1):
        mg.mg_set_density(h, level, -1, delta)
        mg.mg_set_field(h, level, -1, None)  # start from the level below
    mg.mg_solve(h, 0, state["alpha"], state["kappa"], TOL)
    return [_field_and_force(h, level, d)
            for level, d in enumerate([state["delta"], *state["levels"]])]


# ---------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------
#: operations of one cell update or residual of the operator (FMA = 2, sqrt = 1)
_CELL_FLOPS = 38
#: V-cycles that a solve to 1e-8 takes at a contraction of 0.1 per cycle
_CYCLES = 9


def _solve_work(cells, sweeps):
    return {"bytes": 6 * 8 * cells, "flops": _CYCLES * (sweeps + 1) * _CELL_FLOPS * cells * 8 // 7}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        sizes = [n for n in (32, 64, 96, 128) if n <= case["largest"]]
        cells = sum(sizes[k % len(sizes)] ** 3 for k in range(case["count"]))
        return {**_solve_work(cells, 4), "bytes": 3 * 8 * cells}
    cells = case["n"] ** 3
    if kind == "residual":
        return {"bytes": (3 + case["rhs"]) * 8 * cells, "flops": _CELL_FLOPS * cells}
    if kind == "smooth":
        return {"bytes": (3 + case["rhs"]) * 8 * cells,
                "flops": case["sweeps"] * _CELL_FLOPS * cells}
    if kind == "transfer":
        # fine read twice and written once, three coarse arrays of an eighth
        return {"bytes": 3 * 8 * cells + 3 * cells, "flops": 20 * cells + cells}
    if kind == "deposit":
        particles, weights = case["side"] ** 3, 27 if case["scheme"] == 2 else 8
        return {"bytes": (3 if case["equal_mass"] else 4) * 8 * particles + 8 * cells,
                "flops": particles * (3 * weights + 20)}
    cells += 512 * (case.get("patches", 0) + case.get("patches", 0) // 32)
    return _solve_work(cells, case.get("nu_pre", 2) + case.get("nu_post", 2))


# ---------------------------------------------------------------------------
# The same in plain torch
# ---------------------------------------------------------------------------
def _stencil(phi):
    def at(dz, dy, dx):
        return torch.roll(phi, (-dz, -dy, -dx), (0, 1, 2))

    sx, sy, sz = at(0, 0, 1) + at(0, 0, -1), at(0, 1, 0) + at(0, -1, 0), at(1, 0, 0) + at(-1, 0, 0)
    cxy = at(0, 1, 1) + at(0, -1, -1) - at(0, -1, 1) - at(0, 1, -1)
    cxz = at(1, 0, 1) + at(-1, 0, -1) - at(-1, 0, 1) - at(1, 0, -1)
    cyz = at(1, 1, 0) + at(-1, -1, 0) - at(-1, 1, 0) - at(1, -1, 0)
    quad = ((sx - sy) ** 2 + (sx - sz) ** 2 + (sy - sz) ** 2) / 3
    quad += (cxy ** 2 + cxz ** 2 + cyz ** 2) / 8
    return sx + sy + sz, quad


def _source(delta, alpha, kappa, floor):
    """1 + 4(1-w) alpha kappa delta, held at 0 from below with the source floor."""
    src = 1.0 + 8.0 / 3.0 * alpha * kappa * delta
    return src.clamp_min(0.0) if floor else src


def _root(quad, src, delta, alpha, kappa, n):
    if alpha == 0.0:
        return kappa * delta
    c3 = 8.0 / 3.0 * alpha
    q = src + c3 * alpha * float(n) ** 4 * quad
    return 2.0 / c3 * (q.clamp_min(0.0).sqrt() - 1.0)


def _exact_residual(delta, phi, rhs, alpha, kappa):
    n = phi.shape[0]
    face, quad = _stencil(phi)
    src = _source(delta, alpha, kappa, False)
    d = (face - 6.0 * phi) * float(n * n) - _root(quad, src, delta, alpha, kappa, n)
    if rhs is not None:
        d -= rhs
    return [d, float(d.max()), float(d.min()), None, None]


def _exact_smooth(case, delta, phi, rhs, alpha, kappa):
    n = phi.shape[0]
    src = _source(delta, alpha, kappa, False)
    r = torch.arange(n, device=phi.device)
    kz, jy, ix = r[:, None, None], r[None, :, None], r[None, None, :]
    colour = ((ix + kz) & 1) + 2 * ((jy + kz) & 1)
    target = 0.01 if rhs is None else rhs + 0.01
    for _ in range(case["sweeps"]):
        for c in range(4):
            face, quad = _stencil(phi)
            new = face - (_root(quad, src, delta, alpha, kappa, n) + target) / float(n * n)
            phi = torch.where(colour == c, new / 6.0, phi)
    return phi


def _exact_transfer(state):
    fine = state["fine"]
    h = fine.shape[0] // 2
    corr = state["coarse"] - state["coarse_ref"]
    for axis in range(3):
        lo, hi = corr.roll(1, axis), corr.roll(-1, axis)
        corr = torch.stack((0.25 * lo + 0.75 * corr, 0.75 * corr + 0.25 * hi), dim=axis + 1)
        corr = corr.flatten(axis, axis + 1)
    return [fine.reshape(h, 2, h, 2, h, 2).mean(dim=(1, 3, 5)), fine + corr]


def _exact_deposit(case, state):
    n, pos = case["n"], state["pos"]
    mass = state["mass"] if state["mass"] is not None else 1.0 / pos.shape[1]
    rho = torch.zeros(n ** 3, dtype=torch.float64, device=pos.device)
    base, weights = [], []
    for a in range(3):
        s = pos[a] * n - 0.5
        if case["scheme"] == 2:
            c = torch.floor(s + 0.5)
            d = s - c
            base.append(c.long() - 1)
            weights.append((0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2))
        else:
            c = torch.floor(s)
            base.append(c.long())
            weights.append((1.0 - (s - c), s - c))
    for k, wz in enumerate(weights[2]):
        for j, wy in enumerate(weights[1]):
            for i, wx in enumerate(weights[0]):
                cell = (((base[2] + k) % n) * n + (base[1] + j) % n) * n + (base[0] + i) % n
                rho.index_add_(0, cell, wx * wy * wz * mass * float(n) ** 3)
    return rho.reshape(n, n, n) - 1.0


def _exact_field(delta, alpha, kappa, depth=6, most=300):
    """The solution of L phi = mean(L phi), mean(phi) = 0: each step solves the Laplacian of
    the residual by FFT, with Anderson's extrapolation over the last `depth` steps."""
    n = delta.shape[0]
    if alpha == 0.0:
        return _poisson(kappa * delta)
    src = _source(delta, alpha, kappa, True)
    phi, xs, gs = torch.zeros_like(delta), [], []
    best, best_phi, worse = math.inf, phi, 0
    for _ in range(most):
        face, quad = _stencil(phi)
        d = (face - 6.0 * phi) * float(n * n) - _root(quad, src, delta, alpha, kappa, n)
        d -= d.mean()
        res = float(d.abs().max())
        worse = 0 if res < 0.9 * best else worse + 1
        if res < best:
            best, best_phi = res, phi
        if worse > 12:
            break
        g = -_poisson(d)
        xs, gs = (xs + [phi])[-depth:], (gs + [g])[-depth:]
        phi = phi + g
        if len(xs) > 1:
            dg = [b - a for a, b in zip(gs, gs[1:])]
            m = torch.tensor([[float((a * b).sum()) for b in dg] for a in dg], dtype=torch.float64)
            v = torch.tensor([float((a * g).sum()) for a in dg], dtype=torch.float64)
            m += 1e-14 * m.diagonal().max() * torch.eye(len(dg), dtype=torch.float64)
            for w, a, b, e in zip(torch.linalg.solve(m, v).tolist(), xs, xs[1:], dg):
                phi = phi - w * ((b - a) + e)
    return best_phi - best_phi.mean()


def _exact_force(phi):
    s = -0.25 * phi.shape[0]
    return torch.stack([s * (phi.roll(-1, a) - phi.roll(1, a)) for a in (2, 1, 0)])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("residual", "smooth"):
        delta, phi, rhs, alpha, kappa = _field_inputs(case, seed)
        if kind == "residual":
            return _exact_residual(delta, phi, rhs, alpha, kappa)
        return _exact_smooth(case, delta, phi, rhs, alpha, kappa)
    if kind == "batch":
        return [_exact_field(inputs.lognormal_delta_device(s["n"], s["sigma"], seed + k),
                             s["alpha"], s["kappa"])
                for k, s in enumerate(_batch_specs(case, seed))]
    if kind in ("solve", "refined"):
        alpha, kappa = _parameters(case)
        phi = _exact_field(inputs.lognormal_delta_device(case["n"], case["sigma"], seed), alpha,
                           kappa)
        out = [phi, _exact_force(phi)]
        # the patches of the refinement levels have no such short form
        return out if kind == "solve" else [out, None, None]
    state = prepare(case, seed)
    return _exact_transfer(state) if kind == "transfer" else _exact_deposit(case, state)
