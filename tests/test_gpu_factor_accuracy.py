"""Accuracy of the 16-column factorisation at the largest blocks: its rank-16
updates are summed before they meet the matrix entries, one rounding a panel, so
an unrefined solve is about as accurate as with the slab form's rank-128 updates.

The bar, twice the slab form's residual of the same solve, allows for the
48 updates of an entry against 6 and for the other pivot order; sixteen
roundings a panel against the entries gave three times that residual.
"""
import pytest

import workloads as W
from tests.gpu_util import lib, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0, 1, 2])
@pytest.mark.parametrize("adjoint", [False, True])
def test_unrefined_residual_against_the_slab_form(seed, adjoint):
    torch = torch_cuda()
    rr = lib()
    g = W.ns_grid(24, 256)
    o = rr.Operator(g, W.smooth_random_flow(g, seed))
    gen = torch.Generator(device="cuda:0").manual_seed(seed)
    b = torch.randn(2, o.n, 16, dtype=torch.complex128, device="cuda:0", generator=gen)
    res = {}
    for precision in ("fp32", "fp32_simt"):
        fa = o.factor([0.05 + 0.4j, 0.05 + 2.5j], precision)
        _, info = fa.solve(b, adjoint, refine_tol=0.0, max_refine=0, check=False)
        res[precision] = info["first_residual"]
        fa.close()
    assert res["fp32_simt"] <= 2.0 * res["fp32"]
    o.close()
