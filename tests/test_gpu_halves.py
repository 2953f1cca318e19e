"""GPU parity where the two halves of the factorisation and of the sweeps meet:
the fewest columns (one on each side of the middle), halves of equal and of
unequal length, in every form: FP64 and FP32 in the cluster sweeps, and the
batched tensor-core sweeps with the slab factorisation.

Checked against the oracle's dense LU solve on the same inputs with the bars of
the solve tests (FP64 1e-11, FP32 with refinement 1e-9).
"""
import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from tests.gpu_util import lib, rel_err, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [3, 4, 5, 8])
@pytest.mark.parametrize("ny,k,F,precision", [(11, 3, 2, "fp64"), (11, 3, 2, "fp32"),
                                              (48, 16, 40, "fp32")])
@pytest.mark.parametrize("adjoint", [False, True])
def test_halves_meet(nx, ny, k, F, precision, adjoint):
    torch = torch_cuda()
    rr = lib()
    g = W.ns_grid(nx, ny)
    flow = W.smooth_random_flow(g, 33)
    L = op.assemble(g, flow)
    o = rr.Operator(g, flow)
    shifts = 0.05 + 1j * np.linspace(0.4, 2.5, F)
    fa = o.factor(shifts, precision)
    rng = np.random.default_rng(nx * 10 + k)
    b = rng.standard_normal((F, o.n, k)) + 1j * rng.standard_normal((F, o.n, k))
    x, _ = fa.solve(to_dev(b, torch), adjoint, refine_tol=1e-12, max_refine=20)
    for f in (0, F - 1):
        A = op.shifted(L, shifts[f]).toarray()
        want = np.linalg.solve(A.conj().T if adjoint else A, b[f])
        assert rel_err(x[f].cpu().numpy(), want) < (1e-11 if precision == "fp64" else 1e-9)
    fa.close()
    o.close()
