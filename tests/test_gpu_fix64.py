"""Smoothing stages in tiles and cell by cell, on fields whose values need every path of the
integer arithmetic, against the same sweep in extended precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1303_0008_gb300 import mg  # noqa: E402

Q = np.longdouble
ALPHA, KAPPA, LAM = 0.3, 1.0, 0.01


def forms(p):
    def at(dz, dy, dx):
        return np.roll(p, (-dz, -dy, -dx), (0, 1, 2))

    sx, sy, sz = at(0, 0, 1) + at(0, 0, -1), at(0, 1, 0) + at(0, -1, 0), at(1, 0, 0) + at(-1, 0, 0)
    cxy = at(0, 1, 1) + at(0, -1, -1) - at(0, -1, 1) - at(0, 1, -1)
    cxz = at(1, 0, 1) + at(-1, 0, -1) - at(-1, 0, 1) - at(1, 0, -1)
    cyz = at(1, 1, 0) + at(-1, -1, 0) - at(-1, 1, 0) - at(1, -1, 0)
    quad = ((sx - sy) ** 2 + (sx - sz) ** 2 + (sy - sz) ** 2) / 3
    return sx + sy + sz, quad + (cxy ** 2 + cxz ** 2 + cyz ** 2) / 8


def root(quad, delta, n):
    c3 = Q(8) / 3 * Q(ALPHA)
    q = 1 + c3 * Q(KAPPA) * delta + c3 * Q(ALPHA) * quad * Q(n) ** 4
    return 2 / c3 * (np.sqrt(np.maximum(q, 0)) - 1)


def sweep(phi, delta, f, n):
    p = phi.astype(Q)
    i = np.arange(n)
    colour = (((i[None, None, :] + i[:, None, None]) & 1) +
              2 * ((i[None, :, None] + i[:, None, None]) & 1))
    for c in range(4):
        face, quad = forms(p)
        p = np.where(colour == c, (face - (root(quad, delta, n) + f + Q(LAM)) / (n * n)) / 6, p)
    return p


def field(kind, n, rng):
    x = np.arange(n) / n
    wave = (np.sin(2 * np.pi * x)[:, None, None] * np.cos(4 * np.pi * x)[None, :, None] +
            0.3 * np.sin(6 * np.pi * x)[None, None, :])
    noise = rng.standard_normal((n, n, n))
    return {"one binade": 1.5 + 0.2 * wave, "waves": 0.01 * wave, "noise": 1e-3 * noise,
            "zero": np.zeros((n, n, n)),
            "spikes": np.where(rng.random((n, n, n)) < 1e-3, 1.0, 1e-9) * noise,
            "tiny": 1e-150 * noise}[kind]


@pytest.mark.parametrize("n", [30, 112, 114])
@pytest.mark.parametrize("kind", ["one binade", "waves", "noise", "zero", "spikes", "tiny"])
def test_sweep(n, kind):
    rng = np.random.default_rng(n)
    phi = np.ascontiguousarray(field(kind, n, rng))
    delta = rng.uniform(-0.5, 3.0, (n, n, n))
    f = rng.uniform(-0.1, 0.1, (n, n, n)) if n != 112 else np.zeros((n, n, n))
    out = torch.from_numpy(phi).cuda()
    mg.mg_op_smooth(n, out, torch.from_numpy(delta).cuda(),
                    torch.from_numpy(f).cuda() if n != 112 else None, 0, ALPHA, KAPPA, LAM, 1)
    want = sweep(phi, delta, f, n)
    # an update: a few roundings of terms no larger than the largest value; the four stages
    # pass errors on by a factor of at most 1 + sqrt(2/3) each (the slope of the root)
    scale = max(np.abs(phi).max(), float(np.abs(want).max()))
    tol = 4 * 2.0 ** -53 * scale * 1.82 ** 4
    assert np.abs(out.cpu().numpy() - want).max() <= tol


@pytest.mark.parametrize("n", [66, 114])
@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e200])
def test_values_without_an_integer_form(n, bad):
    """They spread to the cells that read them and to no others."""
    rng = np.random.default_rng(3)
    phi = 1e-3 * rng.standard_normal((n, n, n))
    delta = rng.uniform(-0.5, 3.0, (n, n, n))
    d = torch.from_numpy(delta).cuda()
    a = torch.from_numpy(phi).cuda()
    mg.mg_op_smooth(n, a, d, None, 0, ALPHA, KAPPA, LAM, 1)
    phi[5, 6, 7] = bad
    b = torch.from_numpy(phi).cuda()
    mg.mg_op_smooth(n, b, d, None, 0, ALPHA, KAPPA, LAM, 1)
    a, b = a.cpu().numpy(), b.cpu().numpy()
    far = np.ones(phi.shape, bool)
    far[0:11, 1:12, 2:13] = False  # four stages reach four cells
    assert np.isfinite(a).all() and np.isfinite(b[far]).all()
    assert np.abs(a[far] - b[far]).max() <= 4 * 2.0 ** -53 * np.abs(a).max() * 1.82 ** 4
    if not np.isfinite(bad):
        assert not np.isfinite(b[4:7, 5:8, 6:9]).all()


@pytest.mark.parametrize("n", [112, 128])
@pytest.mark.parametrize("alpha", [0.0, -0.3, 5e-5])
def test_other_modes_in_tiles(n, alpha):
    """The linear and the conjugate form, and the other branch, against one cell at a time
    in extended precision at a few cells of the first colour."""
    rng = np.random.default_rng(7)
    phi = 1e-3 * rng.standard_normal((n, n, n))
    delta = rng.uniform(-0.5, 3.0, (n, n, n))
    kappa = -1.0 if alpha < 0 else 1.0
    out = torch.from_numpy(phi).cuda()
    mg.mg_op_smooth(n, out, torch.from_numpy(delta).cuda(), None, 0, alpha, kappa, LAM, 1)
    face, quad = forms(phi.astype(Q))
    if alpha == 0.0:
        D = kappa * delta.astype(Q)
    else:
        c3 = Q(8) / 3 * Q(alpha)
        u = Q(kappa) * delta + Q(alpha) * quad * Q(n) ** 4
        D = 2 * u / (1 + np.sqrt(np.maximum(1 + c3 * u, 0)))
    want = (face - (D + Q(LAM)) / (n * n)) / 6
    i = np.arange(n)
    first = (((i[None, None, :] + i[:, None, None]) & 1) == 0) & \
        (((i[None, :, None] + i[:, None, None]) & 1) == 0)
    got = out.cpu().numpy()
    # k2 (sqrt q - 1) loses eps k2 to cancellation
    k2 = 0.0 if abs(alpha) < 1e-4 else abs(2 / (8 / 3 * alpha))
    tol = 8 * 2.0 ** -53 * (np.abs(phi).max() + float(np.abs(D).max() + k2) / (n * n))
    assert np.abs(got - want)[first].max() <= tol


@pytest.mark.parametrize("mixed", [False, True])
def test_batch_in_tiles_has_the_bits_of_single_grids(mixed):
    """Sides below, at and above the first that runs in tiles."""
    from paper_1303_0008_gb300 import inputs as I

    opt = dict(prec=mg.MG_MIXED if mixed else mg.MG_FP64)
    specs = [(n, I.lognormal_delta(n, 1.5, n), s * I.alpha_kappa_for_rv(8.0), s)
             for n, s in ((96, 1.0), (112, -1.0), (128, 1.0), (160, 1.0))]
    g = mg.mg_create_batch([n for n, *_ in specs], mg.options(**opt))
    try:
        for k, (_, d, _, _) in enumerate(specs):
            mg.mg_set_density(g, 0, k, d)
        mg.mg_solve_batch(g, [0] * len(specs), [a for _, _, a, _ in specs],
                          [s for *_, s in specs], 1e-8)
        batch = [mg.mg_get_field(g, 0, k, np.empty((n,) * 3)) for k, (n, *_) in enumerate(specs)]
    finally:
        mg.mg_destroy_grid(g)
    for (n, d, a, s), got in zip(specs, batch):
        h = mg.mg_create_grid(n, mg.options(**opt))
        try:
            mg.mg_set_density(h, 0, -1, d)
            mg.mg_solve(h, 0, a, s, 1e-8)
            assert np.array_equal(mg.mg_get_field(h, 0, -1, np.empty((n,) * 3)), got)
        finally:
            mg.mg_destroy_grid(h)


@pytest.mark.parametrize("n", [94, 96, 100, 134, 258])
def test_prolongation_by_columns(n):
    """Against the tensor product of (3/4, 1/4), and a field that is not 16-byte aligned,
    which goes cell by cell, bit for bit."""
    rng = np.random.default_rng(n)
    h = n // 2
    c, r = (torch.from_numpy(rng.standard_normal((h, h, h))).cuda() for _ in range(2))
    f = torch.from_numpy(rng.standard_normal((n, n, n))).cuda()
    want = c - r
    for axis in range(3):
        lo, hi = want.roll(1, axis), want.roll(-1, axis)
        want = torch.stack((0.25 * lo + 0.75 * want, 0.75 * want + 0.25 * hi), dim=axis + 1)
        want = want.flatten(axis, axis + 1)
    want = want + f
    got = f.clone()
    mg.mg_op_prolong_correct(n, c, r, got)
    odd = torch.empty(n ** 3 + 1, dtype=torch.float64, device="cuda")[1:].view(n, n, n)
    odd.copy_(f)
    mg.mg_op_prolong_correct(n, c, r, odd)
    torch.cuda.synchronize()
    # three multiply-adds and one more, of values up to max|c - r| and max|f|
    tol = 8 * 2.0 ** -53 * float((c - r).abs().max() + f.abs().max())
    assert float((got - want).abs().max()) <= tol
    assert torch.equal(got, odd)


@pytest.mark.parametrize("n", [32, 48, 128])
def test_force_factor(n):
    """-(n/4) times the difference, rounded once: by the exponent where n is a power of two."""
    rng = np.random.default_rng(n)
    phi = rng.standard_normal((n, n, n)) * np.exp(rng.uniform(-650, 300, (n, n, n)))
    phi[:2] = 0.0
    out = torch.empty((3, n, n, n), dtype=torch.float64, device="cuda")
    mg.mg_op_force(n, torch.from_numpy(phi).cuda(), out)
    torch.cuda.synchronize()
    for a, axis in enumerate((2, 1, 0)):
        want = -0.25 * n * (np.roll(phi, -1, axis) - np.roll(phi, 1, axis))
        assert np.array_equal(out[a].cpu().numpy(), want)
