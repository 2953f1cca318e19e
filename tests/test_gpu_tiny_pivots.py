"""Operators scaled towards the ends of the number range, s I - L times a power of
ten, in the 16-column factorisation (FP64, FP32 on the CUDA cores): a pivot whose square
vanishes is reported as singular, one whose inverse square overflows still gives
the solution, which scales by the inverse power.
"""
import dataclasses

import numpy as np
import pytest

import workloads as W
from oracle import operator as op
from tests.gpu_util import lib, rel_err, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

SINGULAR = 3
G = W.Grid(kind=W.KIND_ADVDIFF, nx=4, ny=20, x0=0, x1=10, y0=-5, y1=5, re=20.0)


def _scaled(c):
    flow = W.smooth_random_flow(G, 3)
    return (dataclasses.replace(G, re=G.re / c),
            W.BaseFlow(rho=flow.rho, u=flow.u * c, v=flow.v * c))


@pytest.mark.parametrize("precision,c", [("fp64", 1e-170), ("fp32_simt", 1e-30)])
def test_vanishing_pivots_are_singular(precision, c):
    torch_cuda()
    rr = lib()
    g, flow = _scaled(c)
    o = rr.Operator(g, flow)
    with pytest.raises(rr.RRError) as e:
        o.factor([(0.05 + 0.8j) * c], precision)
    assert e.value.status == SINGULAR
    o.close()


@pytest.mark.parametrize("precision,c,bar", [("fp64", 1e-150, 1e-11), ("fp64", 1e150, 1e-11),
                                             ("fp64", 3e-158, 1e-6),
                                             ("fp32_simt", 2e-20, 1e-9)])
def test_small_and_large_pivots_solve(precision, c, bar):
    torch = torch_cuda()
    rr = lib()
    flow = W.smooth_random_flow(G, 3)
    L = op.assemble(G, flow)
    gc, fc = _scaled(c)
    o = rr.Operator(gc, fc)
    s = 0.05 + 0.8j
    fa = o.factor([s * c], precision)
    rng = np.random.default_rng(9)
    b = rng.standard_normal((1, o.n, 3)) + 1j * rng.standard_normal((1, o.n, 3))
    x, _ = fa.solve(to_dev(b * c, torch), refine_tol=1e-11, max_refine=20)
    want = np.linalg.solve(op.shifted(L, s).toarray(), b[0])
    assert rel_err(x.cpu().numpy()[0], want) < bar
    fa.close()
    o.close()
