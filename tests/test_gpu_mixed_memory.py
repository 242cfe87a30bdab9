"""Device memory of mixed-precision solves: the finest level's arrays in colour order are left out
where memory is short, with the same result."""
import numpy as np
import pytest

from paper_1303_0008_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1303_0008_gb300 import mg  # noqa: E402


def solve(n, delta, alpha):
    """The field and the device memory that the first solve took."""
    g = mg.mg_create_grid(n, mg.options(prec=mg.MG_MIXED))
    try:
        mg.mg_set_density(g, 0, -1, delta)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        mg.mg_solve(g, 0, alpha, 1.0, 1e-8)
        torch.cuda.synchronize()
        took = before - torch.cuda.mem_get_info()[0]
        return mg.mg_get_field(g, 0, -1, np.empty((n,) * 3)), took
    finally:
        mg.mg_destroy_grid(g)


@pytest.mark.parametrize("n,optional", [(224, True), (256, False)])
def test_colour_order_where_memory_is_short(n, optional):
    delta, alpha = I.lognormal_delta(n, 1.0, 3), I.alpha_kappa_for_rv(4.0)
    solve(n, delta, alpha)  # code and graphs loaded
    phi, took = solve(n, delta, alpha)
    free, total = torch.cuda.mem_get_info()
    assert free > total * 3 // 4
    held = torch.empty(free - total // 2 + (1 << 26), dtype=torch.uint8, device="cuda")
    try:
        phi_short, took_short = solve(n, delta, alpha)
    finally:
        del held
        torch.cuda.empty_cache()
    assert np.array_equal(phi, phi_short)
    arrays = 8 * n ** 3 if optional else 0
    # allocations come in pages of 2 MB; graphs and events take some on the side
    assert abs((took - took_short) - arrays) <= 16 << 20
