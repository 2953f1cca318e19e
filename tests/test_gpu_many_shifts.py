"""More shifts than half a grid dimension holds, in the tensor-core sweeps: both
halves of a solve are one launch, so its problems pass 65,535.

Checked against the oracle's dense LU solve with the FP32 solve bar (1e-9).
"""
import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from tests.gpu_util import lib, rel_err, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("adjoint", [False, True])
def test_solve_with_33000_shifts(adjoint):
    torch = torch_cuda()
    rr = lib()
    if torch.cuda.mem_get_info()[0] < 90e9:
        pytest.skip("needs 90 GB of device memory")
    from paper_1902_01458_gb300 import _lib
    g = W.Grid(kind=W.KIND_ADVDIFF, nx=3, ny=128, x0=0, x1=10, y0=-5, y1=5, re=20.0)
    flow = W.smooth_random_flow(g, 32)
    L = op.assemble(g, flow)
    o = rr.Operator(g, flow)
    F, k = 33000, 2
    shifts = 0.05 + 1j * np.linspace(0.4, 2.5, F)
    fa = o.factor(shifts, "fp32")
    rng = np.random.default_rng(7)
    b = rng.standard_normal((o.n, k)) + 1j * rng.standard_normal((o.n, k))
    bd = to_dev(b, torch).expand(F, o.n, k).contiguous()
    _lib.rr_profile_start(["sweep"])
    fa.solve(bd, adjoint, refine_tol=0.0, max_refine=0, check=False)
    launches = _lib.rr_profile_read("sweep")[1]
    _lib.rr_profile_start([])
    assert launches == 4  # three products and the middle (the cluster form has two)
    x, _ = fa.solve(bd, adjoint)
    for f in (0, F // 2, F - 1):
        A = op.shifted(L, shifts[f]).toarray()
        want = np.linalg.solve(A.conj().T if adjoint else A, b)
        assert rel_err(x[f].cpu().numpy(), want) < 1e-9
    fa.close()
    o.close()
