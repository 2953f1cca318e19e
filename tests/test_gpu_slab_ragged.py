"""GPU parity of the slab factorisation where one CTA holds a whole problem and its
last panel has eight columns: 104 rows leave nine update warps, more than the
panel has pivots (the rows of B beyond them are cleared while the panel warps
still read the panel before), with 72, 88 and 120 rows on either side of it.

Checked against the oracle's dense LU solve: the unrefined solve to 1e-4
relative (FP32-level factors), the refined one to 1e-9.
"""
import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from tests.gpu_util import lib, rel_err, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q,ny,F", [(1, 104, 24), (1, 104, 140), (4, 26, 80), (1, 72, 40),
                                    (1, 88, 40), (1, 120, 40)])
def test_one_cta_slab_with_a_ragged_panel(q, ny, F):
    torch = torch_cuda()
    rr = lib()
    g = W.kz_grid(3, ny, 0.8) if q == 4 else W.Grid(kind=W.KIND_ADVDIFF, nx=3, ny=ny, x0=0,
                                                    x1=10, y0=-5, y1=5, re=20.0)
    flow = W.smooth_random_flow(g, 21)
    L = op.assemble(g, flow)
    o = rr.Operator(g, flow)
    shifts = 0.02 + 1j * np.linspace(0.2, 4.0, F)
    fa = o.factor(shifts, "fp32")
    rng = np.random.default_rng(ny + F)
    b = rng.standard_normal((F, o.n, 4)) + 1j * rng.standard_normal((F, o.n, 4))
    bd = to_dev(b, torch)
    for _ in range(3):
        fa.refactor(shifts)
        x0, _ = fa.solve(bd, refine_tol=0.0, max_refine=0, check=False)
        x, _ = fa.solve(bd)
        for f in sorted({0, F // 2, F - 1}):
            want = np.linalg.solve(op.shifted(L, shifts[f]).toarray(), b[f])
            assert rel_err(x0[f].cpu().numpy(), want) < 1e-4
            assert rel_err(x[f].cpu().numpy(), want) < 1e-9
    fa.close()
    o.close()
