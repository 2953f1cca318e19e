"""GPU parity of the tensor-core form of the sweeps over what it serves: odd blocks and
numbers of right-hand sides, every operand split, tiles cut by the edge, both directions.  Each
case is a batch that takes this form (its launches are counted: one per column
pair and direction, where the cluster form has two in all).

Checked against the oracle's dense LU solve: the refined solve to 1e-9, and the
unrefined one to the bars of the factors, 1e-4 (BF16x3, 16 bits a product: 1e-2).
"""
import dataclasses

import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from tests.gpu_util import lib, rel_err, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def check(kind, nx, ny, k, F, precision, periodic=False, adjoint=False):
    torch = torch_cuda()
    rr = lib()
    from paper_1902_01458_gb300 import _lib
    if kind == "kz":
        g = W.kz_grid(nx, ny, 0.8)
    elif kind == "ns":
        g = W.ns_grid(nx, ny)
    else:
        g = W.Grid(kind=W.KIND_ADVDIFF, nx=nx, ny=ny, x0=0, x1=10, y0=-5, y1=5, re=20.0)
    if periodic:
        g = dataclasses.replace(g, periodic_y=True, sponge_max=0.0)
    flow = W.smooth_random_flow(g, 32)
    L = op.assemble(g, flow)
    o = rr.Operator(g, flow)
    shifts = 0.05 + 1j * np.linspace(0.4, 2.5, F)
    fa = o.factor(shifts, precision)
    rng = np.random.default_rng(ny * 10 + k)
    b = rng.standard_normal((F, o.n, k)) + 1j * rng.standard_normal((F, o.n, k))
    bd = to_dev(b, torch)
    _lib.rr_profile_start(["sweep"])
    x0, _ = fa.solve(bd, adjoint, refine_tol=0.0, max_refine=0, check=False)
    launches = _lib.rr_profile_read("sweep")[1]
    _lib.rr_profile_start([])
    assert launches == 2 * (nx // 2) + 2  # the products and the middle column's
    x, _ = fa.solve(bd, adjoint)
    for f in sorted({0, F // 2, F - 1}):
        A = op.shifted(L, shifts[f]).toarray()
        want = np.linalg.solve(A.conj().T if adjoint else A, b[f])
        assert rel_err(x0[f].cpu().numpy(), want) < (1e-2 if precision.endswith("x3") else 1e-4)
        assert rel_err(x[f].cpu().numpy(), want) < 1e-9
    fa.close()
    o.close()


@pytest.mark.parametrize("kind,ny,k,F,precision,periodic",
                         [("ns", 128, 15, 32, "fp32", False), ("ns", 256, 1, 16, "fp32", False),
                          ("ns", 64, 63, 24, "fp32", True), ("kz", 40, 33, 24, "fp32", True),
                          ("ns", 128, 31, 32, "fp32_bf16x3", False),
                          ("ns", 86, 15, 64, "fp32_bf16x6", True)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_odd_columns(kind, ny, k, F, precision, periodic, adjoint):
    check(kind, 5, ny, k, F, precision, periodic, adjoint)


@pytest.mark.parametrize("kind,ny,k,F,precision,periodic",
                         [("ns", 129, 32, 32, "fp32", False), ("ns", 129, 31, 32, "fp32", True),
                          ("ns", 129, 64, 24, "fp32", False), ("ad", 341, 9, 40, "fp32", True),
                          ("ns", 85, 9, 64, "fp32_bf16x6", False),
                          ("ns", 129, 16, 40, "fp32_bf16x3", True)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_odd_blocks(kind, ny, k, F, precision, periodic, adjoint):
    """Rows of G, and with odd k the right-hand sides, do not start on 16 bytes."""
    check(kind, 5, ny, k, F, precision, periodic, adjoint)


@pytest.mark.parametrize("kind,ny,k,F,precision,periodic",
                         [("ns", 42, 32, 64, "fp32", False), ("ns", 21, 63, 96, "fp32", True),
                          ("kz", 12, 64, 128, "fp32", False), ("kz", 31, 32, 64, "fp32_bf16x3", True),
                          ("ns", 32, 32, 96, "fp32_bf16x6", False)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_blocks_smaller_than_a_tile(kind, ny, k, F, precision, periodic, adjoint):
    check(kind, 5, ny, k, F, precision, periodic, adjoint)


@pytest.mark.parametrize("kind,ny,k,F", [("ns", 128, 16, 40), ("ns", 130, 32, 24),
                                         ("ad", 130, 32, 96)])
@pytest.mark.parametrize("precision", ["fp32", "fp32_bf16x3", "fp32_bf16x6"])
@pytest.mark.parametrize("adjoint", [False, True])
def test_operand_splits(kind, ny, k, F, precision, adjoint):
    check(kind, 5, ny, k, F, precision, False, adjoint)


@pytest.mark.parametrize("ny,k,F", [(128, 64, 24), (129, 33, 32)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_bf16x6_beyond_32_columns(ny, k, F, adjoint):
    check("ns", 5, ny, k, F, "fp32_bf16x6", False, adjoint)


@pytest.mark.parametrize("ny,k,F", [(64, 8, 32), (64, 7, 64), (16, 4, 128)])
def test_small_batches_stay_in_the_cluster_form(ny, k, F):
    """Two launches a solve: the form that measured faster there."""
    torch = torch_cuda()
    rr = lib()
    from paper_1902_01458_gb300 import _lib
    g = W.ns_grid(9, ny)
    o = rr.Operator(g, W.smooth_random_flow(g, 32))
    fa = o.factor(0.05 + 1j * np.linspace(0.4, 2.5, F), "fp32")
    b = torch.ones(F, o.n, k, dtype=torch.complex128, device="cuda:0")
    _lib.rr_profile_start(["sweep"])
    fa.solve(b, refine_tol=0.0, max_refine=0, check=False)
    launches = _lib.rr_profile_read("sweep")[1]
    _lib.rr_profile_start([])
    assert launches == 2
    fa.close()
    o.close()


@pytest.mark.parametrize("kind,ny,k,F,periodic", [("ns", 128, 32, 48, False), ("ns", 129, 16, 64, True),
                                                  ("ad", 257, 63, 32, False), ("kz", 33, 64, 64, True),
                                                  ("ns", 256, 16, 48, False)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_cuda_core_product(kind, ny, k, F, periodic, adjoint):
    """Large batches of FP32 factors without tensor cores take the same form."""
    check(kind, 5, ny, k, F, "fp32_simt", periodic, adjoint)


@pytest.mark.parametrize("seed", [0, 1, 2])
@pytest.mark.parametrize("adjoint", [False, True])
def test_sixty_four_columns_are_as_accurate_as_thirty_two(seed, adjoint):
    """The same 32 right-hand sides twice: both widths sum hi.hi in two accumulators over
    equally long parts of the contraction, so the unrefined residuals agree up to the
    small orders; a tenth is allowed (one accumulator rounds towards zero twice as often)."""
    torch = torch_cuda()
    rr = lib()
    g = W.ns_grid(24, 128)
    o = rr.Operator(g, W.smooth_random_flow(g, seed))
    F = 24
    fa = o.factor(0.05 + 1j * np.linspace(0.4, 2.5, F), "fp32")
    gen = torch.Generator(device="cuda:0").manual_seed(seed)
    b = torch.randn(F, o.n, 32, dtype=torch.complex128, device="cuda:0", generator=gen)
    res = [fa.solve(v, adjoint, refine_tol=0.0, max_refine=0, check=False)[1]["first_residual"]
           for v in (b, torch.cat([b, b], dim=2))]
    assert res[1] <= 1.1 * res[0]
    fa.close()
    o.close()
