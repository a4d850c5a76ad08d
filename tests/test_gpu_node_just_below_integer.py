"""Nodes whose Re w lies so little below an integer that Re w - floor(Re w) rounds to
1: they are nodes at that integer to within the rounding of the phase, in the
product and in the adjoint, on sparse and dense grids and in direct sums."""
import numpy as np
import pytest

import oracle
from paper_1606_03255_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def fl():
    from paper_1606_03255_gb300 import build as libbuild
    libbuild.build()
    from paper_1606_03255_gb300 import fl as flmod
    flmod.load()
    return flmod


@pytest.mark.parametrize("prec,eps", [("fp32", 1e-6), ("fp64", 1e-10), ("fp64ff", 1e-10)])
@pytest.mark.parametrize("route", ["nfft", "direct"])
@pytest.mark.parametrize("N,M", [(40, 3000), (300, 5000), (5000, 200)])    # dense by CTA, by warp, sparse
def test_just_below_an_integer(fl, prec, eps, route, N, M):
    cdt = torch.complex64 if prec == "fp32" else torch.complex128
    w = W.nodes_circle_clustered(M, seed=N)
    w[::2, 0] = -np.array([1e-20, 1e-300, 5e-324, 2.0 ** -55])[np.arange((M + 1) // 2) % 4]
    c, r = W.coefficients(N, seed=1), W.coefficients(M, seed=2)
    dev = torch.device("cuda")
    plan = fl.Plan(N, torch.from_numpy(w).to(dev), eps, precision=prec, route=route)
    f = plan.execute(torch.from_numpy(c).to(cdt).to(dev)).cpu().numpy().astype(np.complex128)
    g = plan.adjoint(torch.from_numpy(r).to(cdt).to(dev)).cpu().numpy().astype(np.complex128)
    plan.close()
    near = w.copy()
    near[::2, 0] = 0.0                                     # k |Re w| < 2^-42
    for got, ref, x in ((f, oracle.flt_direct(c, near), c), (g, oracle.flt_adjoint(r, near, N), r)):
        bound = eps if prec != "fp32" else eps + 32 * U32 * np.max(np.abs(ref)) / np.sum(np.abs(x))
        assert oracle.error_E(ref, got, x) <= bound
