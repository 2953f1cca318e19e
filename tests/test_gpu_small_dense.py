"""GPU parity of the small dense kernels (Gram sums, Cholesky factor and inverse,
triangular and general right products, cluster Jacobi SVD) over the column
counts where their splits change: odd k (a padded column), one warp and several,
one CTA and clusters of two to eight, pair counts that do not divide among the
CTAs.  Algorithm 1 against the oracle with the FP64 bars of the parity tests.
"""
import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from oracle import resolvent as rs
from tests.gpu_util import lib, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 5, 9, 16, 17, 24, 31, 33, 40, 47, 63])
def test_algorithm1_over_column_counts(k):
    torch = torch_cuda()
    rr = lib()
    wl = W.config_small_ns(14, 12, k=k, nfreq=2)
    g, flow = wl.grid, wl.flow
    L = op.assemble(g, flow)
    o = rr.Operator(g, flow)
    shifts = 1j * wl.omegas
    fa = o.factor(shifts, "fp64")
    res = fa.randomized_resolvent(k, [3, 4], orthogonalize=True)
    for f, s in enumerate(shifts):
        ref = rs.randomized(L, s, k, 3 + f, orthogonalize=True)
        np.testing.assert_allclose(res.sigma_halko[f].cpu().numpy(), ref.sigma_halko, rtol=1e-9)
        np.testing.assert_allclose(res.sigma[f].cpu().numpy(), ref.sigma, rtol=1e-9)
        V = res.V[f].cpu().numpy()
        np.testing.assert_allclose(V.conj().T @ V, np.eye(k), atol=1e-12)
        assert rs.principal_angle(V, ref.V) <= 1e-5
    fa.close()
    o.close()
