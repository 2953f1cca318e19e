"""GPU parity of the block sweeps at the sizes where their forms change: rows per
CTA and cluster sizes (one point per CTA up to 129 rows), odd blocks (8-byte
copies), k that does not fill a column group, one, three and four unknowns per
point, periodic y (halos that wrap), FP64 and FP32, both directions; and the
two-launch tensor-core form, which large batches take, with tiles cut by the
edge.

Checked against the oracle's dense LU solve on the same inputs with the bars of
the solve tests (FP64 1e-11, FP32 with refinement 1e-9).
"""
import dataclasses

import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from tests.gpu_util import lib, rel_err, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _grid(kind, nx, ny, periodic):
    if kind == "kz":
        g = W.kz_grid(nx, ny, 0.8)
    elif kind == "ns":
        g = W.ns_grid(nx, ny)
    else:
        g = W.Grid(kind=W.KIND_ADVDIFF, nx=nx, ny=ny, x0=0, x1=10, y0=-5, y1=5, re=20.0)
    return dataclasses.replace(g, periodic_y=True, sponge_max=0.0) if periodic else g


# kind, nx, ny, k, shifts, periodic
CASES = [("ns", 4, 3, 1, 1, False), ("ns", 5, 9, 5, 3, False), ("ns", 4, 17, 11, 2, True),
         ("ad", 6, 5, 3, 2, True), ("ad", 3, 131, 2, 1, False), ("ad", 4, 64, 17, 2, False),
         ("kz", 4, 7, 6, 2, False), ("kz", 3, 40, 9, 1, False), ("ns", 3, 64, 33, 2, False),
         ("ns", 3, 129, 4, 1, False), ("ns", 3, 341, 7, 1, False)]


@pytest.mark.parametrize("kind,nx,ny,k,F,periodic", CASES)
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("adjoint", [False, True])
def test_sweeps_match_oracle(kind, nx, ny, k, F, periodic, precision, adjoint):
    torch = torch_cuda()
    rr = lib()
    g = _grid(kind, nx, ny, periodic)
    flow = W.smooth_random_flow(g, 31)
    L = op.assemble(g, flow)
    o = rr.Operator(g, flow)
    shifts = 0.05 + 1j * np.linspace(0.4, 2.5, F)
    fa = o.factor(shifts, precision)
    rng = np.random.default_rng(ny * 10 + k)
    b = rng.standard_normal((F, o.n, k)) + 1j * rng.standard_normal((F, o.n, k))
    x, _ = fa.solve(to_dev(b, torch), adjoint, refine_tol=1e-12, max_refine=20)
    x = x.cpu().numpy()
    for f, s in enumerate(shifts):
        A = op.shifted(L, s).toarray()
        want = np.linalg.solve(A.conj().T if adjoint else A, b[f])
        assert rel_err(x[f], want) < (1e-11 if precision == "fp64" else 1e-9)
    fa.close()
    o.close()


@pytest.mark.parametrize("ny,k,F,precision", [(88, 16, 40, "fp32"), (129, 64, 24, "fp32"),
                                              (45, 6, 160, "fp32_bf16x6"), (130, 32, 24, "fp32")])
@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("adjoint", [False, True])
def test_batched_sweeps_match_oracle(ny, k, F, precision, periodic, adjoint):
    torch = torch_cuda()
    rr = lib()
    g = _grid("ns", 3, ny, periodic)
    flow = W.smooth_random_flow(g, 32)
    L = op.assemble(g, flow)
    o = rr.Operator(g, flow)
    shifts = 0.05 + 1j * np.linspace(0.4, 2.5, F)
    fa = o.factor(shifts, precision)
    rng = np.random.default_rng(ny * 10 + k)
    b = rng.standard_normal((F, o.n, k)) + 1j * rng.standard_normal((F, o.n, k))
    x, _ = fa.solve(to_dev(b, torch), adjoint)
    for f in (0, F - 1):
        A = op.shifted(L, shifts[f]).toarray()
        want = np.linalg.solve(A.conj().T if adjoint else A, b[f])
        assert rel_err(x[f].cpu().numpy(), want) < 1e-9
    fa.close()
    o.close()
