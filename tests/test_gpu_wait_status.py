"""Bounded waits of the sweeps reach the caller as RR_ERR_TIMEOUT in every mode of a
solve.  rr_debug_waits makes the first CTA of the next sweep launch send
nothing, so the waits of its cluster run out with nothing in flight; an ordinary
solve on the same factors in the same process then succeeds.
"""
import ctypes

import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from tests.gpu_util import lib, rel_err, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

TIMEOUT = 6


def _setup(g, shifts, k, precision):
    torch = torch_cuda()
    rr = lib()
    flow = W.smooth_random_flow(g, 2)
    o = rr.Operator(g, flow)
    fa = o.factor(shifts, precision)
    rng = np.random.default_rng(4)
    b = rng.standard_normal((len(shifts), o.n, k)) + 1j * rng.standard_normal((len(shifts), o.n, k))
    return torch, rr, flow, o, fa, b, to_dev(b, torch)


@pytest.mark.parametrize("adjoint", [False, True])
def test_unrefined_fp64_solve_without_info_reports_a_timeout(adjoint):
    """A C caller that asks for one solve and no report: no residual is formed."""
    from paper_1902_01458_gb300 import _lib
    g = W.ns_grid(4, 40)
    torch, rr, flow, o, fa, b, bd = _setup(g, [0.8j], 6, "fp64")
    x = torch.empty_like(bd)

    def solve():
        return _lib.load().rr_solve(fa.handle, 6, int(adjoint), ctypes.c_void_p(bd.data_ptr()),
                                    ctypes.c_void_p(x.data_ptr()), 0.0, 0, None)

    try:
        _lib.rr_debug_waits(2000, 1)
        assert solve() == TIMEOUT
    finally:
        _lib.rr_debug_waits(0, 0)
    assert solve() == 0  # reported once
    A = op.shifted(op.assemble(g, flow), 0.8j).toarray()
    want = np.linalg.solve(A.conj().T if adjoint else A, b[0])
    assert rel_err(x.cpu().numpy()[0], want) < 1e-11
    x2, _ = fa.solve(bd, adjoint, refine_tol=1e-12)
    assert rel_err(x2.cpu().numpy()[0], want) < 1e-11
    fa.close()
    o.close()


@pytest.mark.parametrize("precision,ny,k,F", [("fp32", 128, 16, 40), ("fp32", 129, 15, 40),
                                              ("fp32", 128, 64, 24), ("fp32_bf16x3", 128, 16, 40),
                                              ("fp32_bf16x6", 128, 32, 24)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_tensor_core_sweep_reports_a_timeout(precision, ny, k, F, adjoint):
    """Its first CTA issues no copy and no MMA: copies, splitting, MMAs and the epilogue give
    up in turn, and tensor memory is freed for the launches that follow."""
    from paper_1902_01458_gb300 import _lib
    nx = 5
    shifts = 0.05 + 1j * np.linspace(0.4, 2.5, F)
    g = W.ns_grid(nx, ny)
    torch, rr, flow, o, fa, b, bd = _setup(g, shifts, k, precision)
    _lib.rr_profile_start(["sweep"])
    fa.solve(bd, adjoint, refine_tol=0.0, max_refine=0, check=False)
    launches = _lib.rr_profile_read("sweep")[1]
    _lib.rr_profile_start([])
    assert launches == 2 * (nx // 2) + 2  # (two in the cluster form)
    try:
        _lib.rr_debug_waits(2000, 1)
        with pytest.raises(rr.RRError) as e:
            fa.solve(bd, adjoint)
        assert e.value.status == TIMEOUT and "timed out" in e.value.message
    finally:
        _lib.rr_debug_waits(0, 0)
    x, _ = fa.solve(bd, adjoint)
    for f in (0, F - 1):
        A = op.shifted(op.assemble(g, flow), shifts[f]).toarray()
        want = np.linalg.solve(A.conj().T if adjoint else A, b[f])
        assert rel_err(x[f].cpu().numpy(), want) < 1e-9
    fa.close()
    o.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("adjoint", [False, True])
def test_cluster_sweep_reports_a_timeout(precision, adjoint):
    from paper_1902_01458_gb300 import _lib
    g = W.ns_grid(4, 40)
    torch, rr, flow, o, fa, b, bd = _setup(g, [0.8j], 6, precision)
    _lib.rr_profile_start(["sweep"])
    fa.solve(bd, adjoint, refine_tol=0.0, max_refine=0, check=False)
    launches = _lib.rr_profile_read("sweep")[1]
    _lib.rr_profile_start([])
    assert launches == 2
    try:
        _lib.rr_debug_waits(2000, 1)
        with pytest.raises(rr.RRError) as e:
            fa.solve(bd, adjoint, refine_tol=1e-12)
        assert e.value.status == TIMEOUT
    finally:
        _lib.rr_debug_waits(0, 0)
    x, _ = fa.solve(bd, adjoint, refine_tol=1e-12, max_refine=20)
    A = op.shifted(op.assemble(g, flow), 0.8j).toarray()
    want = np.linalg.solve(A.conj().T if adjoint else A, b[0])
    assert rel_err(x.cpu().numpy()[0], want) < (1e-11 if precision == "fp64" else 1e-9)
    fa.close()
    o.close()
