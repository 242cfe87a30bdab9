"""Residual, restriction and coarse right-hand side in tiles (sides that are no multiple of
a tile among them), and refinement patches whose values need the rare paths of the integer
arithmetic."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1303_0008_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1303_0008_gb300 import mg  # noqa: E402
from test_gpu_fix64 import ALPHA, KAPPA, field, forms, root  # noqa: E402

Q = np.longdouble


@pytest.mark.parametrize("n", [30, 112, 114])
@pytest.mark.parametrize("kind", ["one binade", "waves", "noise", "zero", "spikes", "tiny"])
def test_residual(n, kind):
    rng = np.random.default_rng(n)
    phi = np.ascontiguousarray(field(kind, n, rng))
    delta = rng.uniform(-0.5, 3.0, (n, n, n))
    f = rng.uniform(-0.1, 0.1, (n, n, n)) if n != 112 else np.zeros((n, n, n))
    d = torch.empty((n, n, n), dtype=torch.float64, device="cuda")
    norms = mg.mg_op_residual(n, torch.from_numpy(phi).cuda(), torch.from_numpy(delta).cuda(),
                              torch.from_numpy(f).cuda() if n != 112 else None, 0, ALPHA, KAPPA, d)
    face, quad = forms(phi.astype(Q))
    r = root(quad, delta, n)
    want = (face - 6 * phi.astype(Q)) * (n * n) - r - f
    got = d.cpu().numpy()
    # a few roundings of the Laplacian's terms, of sqrt(q) times 2 / c3 and of the results
    tol = 4 * 2.0 ** -53 * (12 * np.abs(phi).max() * n * n + float(np.abs(r).max())
                            + 4 / (8 / 3 * ALPHA) + 0.1)
    assert np.abs(got - want).max() <= tol
    assert norms["max"] == got.max() and norms["min"] == got.min()
    assert norms["guards"] == 0 and norms["nonfinite"] == 0
    # n^3 additions in any order
    assert abs(norms["sum"] - got.sum()) <= 1e-12 * np.abs(got).sum() + 1e-300


@pytest.mark.parametrize("rv", [0.0, 8.0])
def test_restriction_and_coarse_rhs(rv):
    """tau of the first coarse right-hand side, against the oracle's operators at the field
    returned: the solve stops at the check that forms it."""
    n = 224
    delta = I.lognormal_delta(n, 1.5, 77)
    alpha = I.alpha_kappa_for_rv(rv) if rv else 0.0
    g = mg.mg_create_grid(n, mg.options(tau_stop=1.0 / 3.0, max_cycles=60))
    try:
        mg.mg_set_density(g, 0, -1, delta)
        st = mg.mg_solve(g, 0, alpha, 1.0, 1e-14)
        phi = mg.mg_get_field(g, 0, -1, np.empty((n,) * 3))
    finally:
        mg.mg_destroy_grid(g)
    fl, _ = O.density_floor(delta, alpha, 1.0)
    dh, _ = O.residual(phi, fl, alpha, 1.0)
    dH, _ = O.residual(O.restrict(phi), O.restrict(fl), alpha, 1.0)
    tau = dH - O.restrict(dh)
    want = np.abs(tau - tau.mean()).max()
    # the gauge fix after the check moves phi by a constant: roundings of n^2 phi
    assert abs(st["tau"] - want) <= 1e-6 * want


@pytest.mark.parametrize("start", ["zero", "spikes", "tiny"])
def test_patch_values_of_every_path(start):
    """Patches that start from values without a common unit reach the same solution."""
    h = I.refined_hierarchy(16, 2.0, 5, thresholds=(15.0, 40.0))
    L = h["levels"][0]
    alpha = I.alpha_kappa_for_rv(8.0)
    rng = np.random.default_rng(1)
    shape = (len(L["origins"]), 8, 8, 8)
    first = {"zero": np.zeros(shape), "tiny": 1e-160 * rng.standard_normal(shape),
             "spikes": 1e-5 * np.where(rng.random(shape) < 0.01, 1.0, 1e-12)}[start]
    g = mg.mg_create_grid(16, mg.options(patch_mg_levels=1, max_cycles=2000))
    try:
        mg.mg_set_density(g, 0, -1, h["delta0"])
        mg.mg_add_patches(g, 1, L["origins"])
        mg.mg_set_density(g, 1, -1, np.ascontiguousarray(L["delta"]))
        mg.mg_set_field(g, 1, -1, np.ascontiguousarray(first))
        st = mg.mg_solve(g, 0, alpha, 1.0, 1e-11, check=False)
        phi0 = mg.mg_get_field(g, 0, -1, np.empty_like(h["delta0"]))
        phi = mg.mg_get_field(g, 1, -1, np.empty(shape))
    finally:
        mg.mg_destroy_grid(g)
    assert st["rc"] == mg.MG_OK, st
    ref, _ = O.patch_solve(16, 1, L["origins"], L["delta"], phi0, alpha, 1.0, tol=1e-12)
    assert np.abs(phi - ref).max() <= 1e-10 * np.abs(ref).max()
