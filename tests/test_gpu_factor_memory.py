"""Factorisation and solves when device memory does not hold both halves' work
buffers of all problems: it runs over fewer problems at a time, and gives memory up
to a solve's workspace.  The memory left is set by a filler.

Checked against the oracle's dense LU solve (FP64 1e-11, FP32 refined 1e-9).
"""
import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from tests.gpu_util import lib, rel_err, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _sizes(b, nx, F, prec):
    """Bytes of the factors with their sweep buffers, and of the work buffers (X, M,
    the pivot rows) of one half of all problems."""
    c = 16 if prec == "fp64" else 8
    own = F * nx * b * b * c + F * 128 * b * c + (4 * F * 64 * b * 8 if prec == "fp32" else 0)
    half = F * (2 * b * b + 16 * b) * c + (F * 128 * b * 8 if prec == "fp32" else 0)
    return own, half


@pytest.mark.parametrize("prec,ny,F", [("fp32", 256, 301), ("fp64", 128, 201)])
def test_one_half_of_the_work_buffers(prec, ny, F):
    torch = torch_cuda()
    rr = lib()
    g = W.ns_grid(3, ny)
    flow = W.smooth_random_flow(g, 6)
    L = op.assemble(g, flow)
    o = rr.Operator(g, flow)
    shifts = 0.05 + 1j * np.linspace(0.4, 2.5, F)
    k = 4
    rng = np.random.default_rng(8)
    b = rng.standard_normal((o.n, k)) + 1j * rng.standard_normal((o.n, k))
    bd = to_dev(b, torch).expand(F, o.n, k).contiguous()
    out = torch.empty_like(bd)
    o.factor([0.8j], prec).close()  # kernels loaded
    torch.cuda.empty_cache()
    own, half = _sizes(o.b, 3, F, prec)
    # the workspace of a solve: seven blocks of vectors and small change
    ws = F * o.n * k * (4 * 16 + 3 * (16 if prec == "fp64" else 8)) + 64 * MB
    left = own + half + ws + half // 10
    assert left < own + 2 * half
    filler = torch.empty(max(0, torch.cuda.mem_get_info()[0] - left), dtype=torch.uint8,
                         device="cuda:0")
    fa = o.factor(shifts, prec)
    x, _ = fa.solve(bd, refine_tol=1e-12, max_refine=20)
    fa.refactor(shifts)  # and again, with the buffers that are left
    x, _ = fa.solve(bd, refine_tol=1e-12, max_refine=20)
    del filler
    for f in (0, F // 2, F - 1):
        want = np.linalg.solve(op.shifted(L, shifts[f]).toarray(), b)
        assert rel_err(x[f].cpu().numpy(), want) < (1e-11 if prec == "fp64" else 1e-9)
    fa.close()
    o.close()
    del out
    torch.cuda.empty_cache()
