"""The FP64 kernels in tiles, cell by cell and on patches, on fields that fall off through a
tile: every cell against extended precision within a few roundings of its own stencil's values,
and as a whole no further off than the same expressions in numpy's float64; the restriction's
outputs against its children."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1303_0008_gb300 import build as B  # noqa: E402
from paper_1303_0008_gb300 import mg  # noqa: E402
from test_gpu_fix64 import ALPHA, field, forms  # noqa: E402

Q = np.longdouble
EPS = 2.0 ** -53
C3 = 4 * (1 - 1 / 3) * ALPHA  # as the solver forms it


def falling(kind, n, rng):
    """Noise whose amplitude falls through each tile of 32 x 16 x 8 cells, or a field of
    test_gpu_fix64."""
    i, j = np.arange(n) % 32, (np.arange(n) % 16)[:, None]
    noise = rng.standard_normal((n, n, n))
    if kind == "falling":
        return noise * np.exp(-0.15 * i - 0.1 * j)
    if kind == "steep":
        return noise * np.exp(-0.5 * i - 0.3 * j)
    return field(kind, n, rng)


def around(p, op):
    """op over the six values across each cell's faces."""
    v = [np.roll(p, s, axis) for axis in range(3) for s in (1, -1)]
    out = v[0]
    for x in v[1:]:
        out = op(out, x)
    return out


def evaluate(phi, src, alpha, n, defect):
    """Update, or h^2 times the defect, of every cell in extended precision, without a
    right-hand side; phi periodic, or a block whose outer cells come out meaningless."""
    p, h2 = phi.astype(Q), 1 / Q(n * n)
    if alpha == 0.0:
        face, D = around(p, np.add), src.astype(Q)
    elif alpha < 1e-4:
        face, quad = forms(p)
        u = src + Q(alpha) * Q(n) ** 4 * quad
        D = 2 * u / (1 + np.sqrt(1 + Q(4 * (1 - 1 / 3) * alpha) * u))
    else:
        face, quad = forms(p)
        k2 = 2 / Q(C3)
        D = k2 * np.sqrt(np.maximum(src + Q(C3) * Q(alpha) * Q(n) ** 4 * quad, 0)) - k2
    return face - 6 * p - h2 * D if defect else (face - h2 * D) / 6


def evaluate64(phi, src, alpha, n, defect):
    """The same in float64, with the solver's constants."""
    h2 = (1 / n) * (1 / n)
    if alpha == 0.0:
        face, D, root = around(phi, np.add), src, -h2 / 6 * src
    elif alpha < 1e-4:
        face, quad = forms(phi)
        u = src + alpha / (3 * (h2 * h2)) * (3 * quad)
        D = 2 * u / (1 + np.sqrt(1 + 4 * (1 - 1 / 3) * alpha * u))
        root = -h2 / 6 * D
    else:
        face, quad = forms(phi)
        k2 = 2 / C3
        s = np.sqrt(np.maximum(src + C3 * (alpha / (3 * (h2 * h2))) * (3 * quad), 0))
        D, root = k2 * s - k2, -h2 * k2 / 6 * s + h2 / 6 * k2
    return ((face - 6 * phi) * n * n - D) / (n * n) if defect else face * (1 / 6) + root


def terms(phi, src, alpha, n, defect):
    """The largest term of each cell's update (of h^2 times its defect)."""
    if alpha < 1e-4:
        r = np.abs(np.asarray(evaluate(0 * phi, src, alpha, n, True), float))
        if alpha != 0.0:
            u = src + alpha * float(n) ** 4 * forms(phi)[1]
            r = np.abs(2 * u / (1 + np.sqrt(1 + 8 / 3 * alpha * u))) / (n * n)
    else:
        quad = forms(phi)[1]
        r = 2 / C3 * (1 + np.sqrt(np.maximum(src + C3 * alpha * float(n) ** 4 * quad, 0))) / (n * n)
    face = around(np.abs(phi), np.maximum)
    return np.maximum(np.maximum(face, 6 * np.abs(phi)), r) if defect else np.maximum(face, r) / 6


# Roundings of a cell, in EPS times its largest term T.  Update: six values rounded to a unit
# that is no more than twice a rounding of the largest of them 3, the sum 6, the result 8, the
# root's products and its own rounding 7.  Defect: the six and six times the centre (their unit
# half as large against them) 3.5, the Laplacian 7, its product 7, the result 8, the root 6.5.
CELL = {False: 24, True: 32}


def check(got, want, fp, scale, defect):
    e = np.asarray(np.abs(got - want), float) / (EPS * scale)
    f = np.asarray(np.abs(fp - want), float) / (EPS * scale)
    assert e.max() <= CELL[defect], e.max()
    assert np.sqrt((e * e).mean()) <= np.sqrt((f * f).mean())


def slab(n):
    """Planes -2 ... 17 (extended precision is slow): two layers of tiles and the wrap."""
    return np.arange(-2, 18) % n


def inputs(kind, alpha, n):
    rng = np.random.default_rng(n)
    phi = np.ascontiguousarray(falling(kind, n, rng))
    if alpha < 1e-4:  # no source, which would hide small values
        return phi, np.zeros_like(phi), np.zeros_like(phi)
    delta = rng.uniform(-0.3, 3.0, phi.shape)
    return phi, delta, C3 * delta + 1


CASES = [(k, a) for k in ("falling", "steep", "spikes", "noise") for a in (0.0, 1e-7, ALPHA)]


@pytest.mark.parametrize("n", [30, 112, 114])
@pytest.mark.parametrize("kind,alpha", CASES)
def test_update_of_every_cell(kind, alpha, n):
    """The first colour of a sweep (it reads the other colours' first values)."""
    phi, delta, src = inputs(kind, alpha, n)
    out = torch.from_numpy(phi).cuda()
    mg.mg_op_smooth(n, out, torch.from_numpy(delta).cuda(), None, 0, alpha, 1.0, 0.0, 1)
    k, i = slab(n), np.arange(n)
    first = (((i[None, None, :] + k[:, None, None]) & 1) == 0) & \
        (((i[None, :, None] + k[:, None, None]) & 1) == 0)
    first[[0, -1]] = False
    args = (phi[k], src[k], alpha, n, False)
    check(out.cpu().numpy()[k][first], evaluate(*args)[first], evaluate64(*args)[first],
          terms(*args)[first], False)


@pytest.mark.parametrize("n", [30, 112, 114])
@pytest.mark.parametrize("kind,alpha", CASES)
def test_defect_of_every_cell(kind, alpha, n):
    phi, delta, src = inputs(kind, alpha, n)
    d = torch.empty((n, n, n), dtype=torch.float64, device="cuda")
    mg.mg_op_residual(n, torch.from_numpy(phi).cuda(), torch.from_numpy(delta).cuda(), None, 0,
                      alpha, 1.0, d)
    k, inner = slab(n), slice(1, -1)
    args = (phi[k], src[k], alpha, n, True)
    check((d.cpu().numpy()[k].astype(Q) / (n * n))[inner], evaluate(*args)[inner],
          evaluate64(*args)[inner], terms(*args)[inner], True)


# ---- kernels without an entry point of their own ----
SOURCE = r"""
#include "mg_patch.cu"
using namespace mg;
struct Scratch {
  Partial* part = nullptr;
  LevelScalars* sc = nullptr;
  explicit Scratch(size_t n) { cudaMalloc(&part, n * sizeof(Partial)); cudaMalloc(&sc, sizeof(*sc)); }
  ~Scratch() { cudaFree(part); cudaFree(sc); }
  int read(double* out) {
    LevelScalars h;
    if (cudaMemcpy(&h, sc, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    const double v[5] = {h.sum, h.dmax, h.dmin, (double)h.guards, (double)h.nonfinite};
    for (int k = 0; k < 5; ++k) out[k] = v[k];
    return 0;
  }
};
// residual restriction of an n^3 grid
extern "C" int restriction(int n, const double* phi, const double* src, const double* f,
                           double alpha, double* phi_c, double* phihat_c, double* rd_c,
                           double* norms) {
  Scratch s(partials_needed((long long)n * n * n));
  launch_residual_restrict64(0, n, phi, src, f, make_op64(n, alpha, 1.0, 0), phi_c, phihat_c, rd_c,
                             s.part, s.sc);
  return s.read(norms);
}
// residual restriction of `count` patches, then the colour stage 0 on them
extern "C" int patches(int count, int n, double* phi, const double* src, const double* ghost,
                       const int* nbr, double alpha, double* phi_c, double* phihat_c, double* rd_c,
                       double* norms) {
  Scratch s(count);
  const OpConst64 c = make_op64(n, alpha, 1.0, 0);
  const bool lin = c.mode == OP_LINEAR;
  (lin ? k_patch_residual_restrict_fix<true> : k_patch_residual_restrict_fix<false>)
      <<<count, 128>>>(phi, src, ghost, nbr, c, phi_c, phihat_c, rd_c, s.part);
  launch_finalize(0, s.part, count, 512.0 * count, 0, s.sc);
  (lin ? k_patch_smooth_fix<true> : k_patch_smooth_fix<false>)
      <<<count, 128>>>(phi, src, ghost, nbr, c, 0);
  return s.read(norms);
}
"""


@pytest.fixture(scope="module")
def kernels(tmp_path_factory):
    d = tmp_path_factory.mktemp("kernels")
    src, so = d / "kernels.cu", d / "kernels.so"
    src.write_text(SOURCE)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", str(src), "-o", str(so), B.LIB,
                    "-Xlinker", "-rpath," + os.path.dirname(B.LIB), "-lcudart"], check=True)
    return ctypes.CDLL(str(so))


def ptr(t):
    return ctypes.c_void_p(t.data_ptr() if t is not None else None)


@pytest.mark.parametrize("n", [114, 128])
@pytest.mark.parametrize("kind,alpha", [("falling", ALPHA), ("steep", 0.0), ("spikes", ALPHA),
                                        ("zero", ALPHA), ("tiny", ALPHA), ("waves", 0.0)])
def test_restriction_of_every_cell(kernels, kind, alpha, n):
    """R d and its norms from the residual kernel's defects, R phi from the field."""
    phi, delta, src = inputs(kind, alpha, n)
    rng = np.random.default_rng(1)
    f = rng.uniform(-0.1, 0.1, phi.shape) if n == 114 else None
    dev = [torch.from_numpy(a).cuda() if a is not None else None for a in (phi, src, f, delta)]
    out = [torch.full((n // 2,) * 3, np.nan, dtype=torch.float64, device="cuda") for _ in range(3)]
    norms = (ctypes.c_double * 5)()
    assert kernels.restriction(n, ptr(dev[0]), ptr(dev[1]), ptr(dev[2]), ctypes.c_double(alpha),
                               *(ptr(t) for t in out), norms) == 0
    d = torch.empty_like(dev[0])
    ref = mg.mg_op_residual(n, dev[0], dev[3], dev[2], 0, alpha, 1.0, d)
    d = d.cpu().numpy()

    def mean(a):
        return a.reshape(n // 2, 2, n // 2, 2, n // 2, 2).mean(axis=(1, 3, 5))

    rphi, hat, rd = (t.cpu().numpy() for t in out)
    assert np.array_equal(rphi, hat)
    # eight values: seven additions and the unit of the tile's integers; for the defects also
    # the source, rounded twice instead of once
    assert (np.abs(rphi - mean(phi.astype(Q))) <= 8 * EPS * mean(np.abs(phi))).all()
    root = np.abs(src) if alpha == 0.0 else 2 / C3 * (np.sqrt(np.abs(src)) + 1)
    assert (np.abs(rd - mean(d.astype(Q))) <= 8 * EPS * mean(np.abs(d) + root)).all()
    lim = 8 * EPS * (np.abs(d).max() + root.max())
    assert abs(norms[1] - ref["max"]) <= lim and abs(norms[2] - ref["min"]) <= lim
    assert abs(norms[0] - ref["sum"]) <= 1e-12 * np.abs(d).sum() + 8 * EPS * root.sum()
    assert norms[3] == ref["guards"] and norms[4] == 0


@pytest.mark.parametrize("alpha", [0.0, ALPHA])
@pytest.mark.parametrize("rate", [(0.0, 0.0), (0.5, 0.3), (2.0, 1.5)])
def test_patches_of_every_cell(kernels, rate, alpha):
    """Patches without neighbours, falling off through their block."""
    count, n = 24, 256
    rng = np.random.default_rng(7)
    x = np.arange(10)
    block = rng.standard_normal((count, 10, 10, 10)) * np.exp(-rate[0] * x - rate[1] * x[:, None])
    src = rng.uniform(-1, 3.0, (count, 8, 8, 8)) * (alpha != 0.0)
    if alpha != 0.0:
        src = C3 * np.abs(src) + 0.2
    inner = (slice(1, 9),) * 3
    phi = torch.from_numpy(np.ascontiguousarray(block[(slice(None),) + inner])).cuda()
    before = phi.clone()
    ghost = torch.from_numpy(block.copy()).cuda()
    nbr = torch.full((count, 27), -1, dtype=torch.int32, device="cuda")
    dsrc = torch.from_numpy(src).cuda()
    out = [torch.full((count, 4, 4, 4), np.nan, dtype=torch.float64, device="cuda")
           for _ in range(3)]
    norms = (ctypes.c_double * 5)()
    assert kernels.patches(count, n, ptr(phi), ptr(dsrc), ptr(ghost), ptr(nbr),
                           ctypes.c_double(alpha), *(ptr(t) for t in out), norms) == 0
    got, rd = phi.cpu().numpy(), out[2].cpu().numpy() / (n * n)
    i = np.arange(8)
    first = (((i[None, None, :] + i[:, None, None]) & 1) == 0) & \
        (((i[None, :, None] + i[:, None, None]) & 1) == 0)
    assert np.array_equal(got[:, ~first], before.cpu().numpy()[:, ~first])
    ref = {d: [] for d in (False, True)}
    for b, s in zip(block, src):
        S = np.pad(s, 1, constant_values=1.0)
        for d in ref:
            args = (b, S, alpha, n, d)
            ref[d].append([g(*args)[inner] for g in (evaluate, evaluate64, terms)])
    want, fp, scale = (np.array([r[k] for r in ref[False]]) for k in range(3))
    check(got[:, first], want[:, first], fp[:, first], scale[:, first], False)

    def mean(a):
        return a.reshape(count, 4, 2, 4, 2, 4, 2).mean(axis=(2, 4, 6))

    want, fp, scale = (mean(np.array([r[k] for r in ref[True]])) for k in range(3))
    assert (np.abs(rd - want) <= (CELL[True] + 8) * EPS * scale).all()
