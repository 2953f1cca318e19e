"""GPU parity of the cluster-resident slab factorisation at the sizes where its
split of the rows changes: one CTA per problem (four and two lanes per row),
clusters of two to eight CTAs, rows that do not divide among the CTAs, a last
panel of eight columns, a last slab of one panel, more problems than clusters
resident at once.

Checked against the oracle's dense LU solve on the same inputs with the bars of
the wide factorisation: the unrefined solve to 1e-4 relative (FP32-level
factors), the refined one to 1e-9.
"""
import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from tests.gpu_util import lib, rel_err, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

# (ny, problems): b = 3 ny
CASES = [(24, 1), (24, 140), (40, 60), (48, 1), (64, 20), (64, 40), (64, 140), (88, 3),
         (136, 20), (136, 33), (256, 2)]


@pytest.mark.parametrize("ny,F", CASES)
def test_slab_factor_solves_match_oracle(ny, F):
    torch = torch_cuda()
    rr = lib()
    g = W.ns_grid(3, ny)
    flow = W.smooth_random_flow(g, 21)
    L = op.assemble(g, flow)
    o = rr.Operator(g, flow)
    shifts = 0.02 + 1j * np.linspace(0.2, 4.0, F)
    fa = o.factor(shifts, "fp32")
    rng = np.random.default_rng(ny * 100 + F)
    k = 4
    b = rng.standard_normal((F, o.n, k)) + 1j * rng.standard_normal((F, o.n, k))
    bd = to_dev(b, torch)
    x0, _ = fa.solve(bd, refine_tol=0.0, max_refine=0, check=False)
    x, _ = fa.solve(bd)
    for f in sorted({0, F // 2, F - 1}):
        want = np.linalg.solve(op.shifted(L, shifts[f]).toarray(), b[f])
        assert rel_err(x0[f].cpu().numpy(), want) < 1e-4
        assert rel_err(x[f].cpu().numpy(), want) < 1e-9
    fa.close()
    o.close()
