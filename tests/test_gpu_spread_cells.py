"""Adjoint spreading at the edges of its blocks: grids below and above the 256
cells of a block, windows that wrap around the grid's end, more covering nodes
than one staged tile, empty stretches of cells, bands on both sides of the
sparse/dense rule, one and several right-hand sides; adjoint and transposed
evaluation against the oracle with the bounds of the adjoint tests."""
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


def _x(kind, M, g):
    if kind == "ends":           # around x = 0 (mod 1)
        return (g.normal(0.0, 2e-3, M)) % 1.0
    if kind == "point":          # one cell holds them all
        return 0.4999 + 1e-6 * g.random(M)
    if kind == "blocks":         # on the boundaries of 256-cell blocks of most grids
        return (g.integers(0, 64, M) / 64.0 + g.normal(0.0, 1e-4, M)) % 1.0
    return g.random(M)


@pytest.mark.parametrize("kind", ["ends", "point", "blocks", "uniform"])
@pytest.mark.parametrize("N,M", [(9, 40), (100, 3), (120, 700), (700, 2000), (3000, 60), (9000, 5000)])
@pytest.mark.parametrize("prec,eps", [("fp32", 1e-6), ("fp64", 1e-12), ("fp64ff", 1e-12), ("fp32", 1e-3)])
def test_spread(fl, kind, N, M, prec, eps):
    dev = torch.device("cuda")
    cdt = torch.complex64 if prec == "fp32" else torch.complex128
    g = np.random.default_rng(N * 7 + M)
    w = W.nodes_circle_clustered(M, seed=N)
    w[: M // 2] = W.nodes_disk_uniform(M, seed=M)[: M // 2]
    w[:, 0] = _x(kind, M, g)
    r = W.coefficients(M, seed=3)
    plan = fl.Plan(N, torch.from_numpy(w).to(dev), eps, precision=prec, route="nfft")
    rt = torch.from_numpy(r).to(cdt).to(dev)
    a = plan.adjoint(rt).cpu().numpy().astype(np.complex128)
    b = plan.adjoint(rt).cpu().numpy().astype(np.complex128)
    t = plan.transposed(rt).cpu().numpy().astype(np.complex128)
    plan.close()
    assert np.array_equal(a, b)          # no atomics on this route
    ref = oracle.flt_adjoint(r, w, N)
    bound = eps if prec != "fp32" else eps + 32 * U32 * np.max(np.abs(ref)) / np.sum(np.abs(r))
    assert oracle.error_E(ref, a, r) <= bound
    reft = np.conj(oracle.flt_adjoint(np.conj(r), w, N))
    assert oracle.error_E(reft, t, r) <= bound
