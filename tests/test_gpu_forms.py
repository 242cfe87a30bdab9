"""Forms of the operator that share kernels and lists with the default one: relaxed steps on the
domain and on patches, alpha = 0 and the conjugate form, alone and as members of a batch."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1303_0008_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1303_0008_gb300 import mg  # noqa: E402


def solve(n, delta, alpha, kappa, tol, **opt):
    g = mg.mg_create_grid(n, mg.options(**opt))
    try:
        mg.mg_set_density(g, 0, -1, delta)
        st = mg.mg_solve(g, 0, alpha, kappa, tol)
        return mg.mg_get_field(g, 0, -1, np.empty((n,) * 3)), st
    finally:
        mg.mg_destroy_grid(g)


@pytest.mark.parametrize("n", [32, 96, 112])
def test_relaxed_steps_reach_the_solution(n):
    """The oracle's residual of the field, up to the constant of the periodic box."""
    delta, alpha = I.lognormal_delta(n, 1.0, n), I.alpha_kappa_for_rv(4.0)
    phi, st = solve(n, delta, alpha, 1.0, 1e-9, omega=0.8, max_cycles=200)
    floored, _ = O.density_floor(delta, alpha, 1.0)
    d, _ = O.residual(phi, floored, alpha, 1.0)
    # the residual's own rounding: a few of 12 n^2 max|phi|
    assert np.abs(d - d.mean()).max() <= 1e-9 + 64 * 2.0 ** -53 * 12 * n * n * np.abs(phi).max()
    plain, st1 = solve(n, delta, alpha, 1.0, 1e-9)
    assert st["cycles"] > st1["cycles"]
    assert np.abs(phi - plain).max() <= 1e-8 * np.abs(plain).max()


def test_relaxed_steps_on_patches():
    h = I.refined_hierarchy(16, 2.0, 5, thresholds=(15.0, 40.0))
    L, alpha = h["levels"][0], I.alpha_kappa_for_rv(8.0)
    shape = (len(L["origins"]), 8, 8, 8)
    g = mg.mg_create_grid(16, mg.options(omega_patch=0.8, max_cycles=2000))
    try:
        mg.mg_set_density(g, 0, -1, h["delta0"])
        mg.mg_add_patches(g, 1, L["origins"])
        mg.mg_set_density(g, 1, -1, np.ascontiguousarray(L["delta"]))
        mg.mg_solve(g, 0, alpha, 1.0, 1e-11)
        phi0 = mg.mg_get_field(g, 0, -1, np.empty_like(h["delta0"]))
        phi = mg.mg_get_field(g, 1, -1, np.empty(shape))
    finally:
        mg.mg_destroy_grid(g)
    ref, _ = O.patch_solve(16, 1, L["origins"], L["delta"], phi0, alpha, 1.0, tol=1e-12)
    assert np.abs(phi - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("opt", [dict(), dict(omega=0.8, max_cycles=200), dict(prec=mg.MG_MIXED)])
def test_batch_of_all_forms_has_the_bits_of_single_grids(opt):
    """Sides that go cell by cell, in tiles, or both on their way down; the solves converge at
    different cycles, so that the lists are made again; twice on one handle."""
    a8 = I.alpha_kappa_for_rv(8.0)
    specs = [(32, a8, 1.0), (96, 0.0, 1.0), (96, 5e-5, 1.0), (112, 0.0, 1.0), (112, 5e-5, 1.0),
             (128, -a8, -1.0), (128, 0.0, -1.0), (48, 5e-5, 1.0)]
    deltas = [I.lognormal_delta(n, 1.0, 10 + k) for k, (n, *_) in enumerate(specs)]
    g = mg.mg_create_batch([n for n, *_ in specs], mg.options(**opt))
    try:
        for _ in range(2):
            for k, d in enumerate(deltas):
                mg.mg_set_density(g, 0, k, d)
                mg.mg_set_field(g, 0, k, np.zeros_like(d))
            mg.mg_solve_batch(g, [0] * len(specs), [a for _, a, _ in specs],
                              [s for *_, s in specs], 1e-8)
            got = [mg.mg_get_field(g, 0, k, np.empty_like(d)) for k, d in enumerate(deltas)]
    finally:
        mg.mg_destroy_grid(g)
    for (n, a, s), d, x in zip(specs, deltas, got):
        y = solve(n, d, a, s, 1e-8, **opt)[0]
        if "prec" in opt and a == 0.0 and n & (n - 1):
            # h^2 is no power of two, and the FP32 linear update rounds its product or not as the
            # compiler fuses it in each kernel: the converged FP64 fields agree to the tolerance
            assert np.abs(x - y).max() <= 1e-8 * np.abs(y).max()
        else:
            assert np.array_equal(x, y), (n, a)
