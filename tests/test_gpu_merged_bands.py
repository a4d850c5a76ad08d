"""Neighbouring bands near the circle evaluated together at one rank: forward,
derivative, adjoint, transposed and real-exponent transforms against the oracle
on node sets that fill those bands evenly, sparsely, at their edges and in one
band only, with the bounds of the forward and adjoint tests; and the merged plan
against the unmerged one (route "nfft") at the bound both keep."""
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


def _nodes(kind, N, M, eps, seed):
    """Im w by kind; the bands with l_m = 1 hold y <= about ln(3/eps) * 2 / N."""
    g = np.random.default_rng(seed)
    x, top = g.random(M), 2.0 * np.log(3.0 / eps) / N
    y1 = np.log(1.0 / eps)
    if kind == "octaves":        # even per band, down to y N = 1e-9
        y = top * 10.0 ** (-10.0 * g.random(M))
    elif kind == "uniform":
        y = top * g.random(M)
    elif kind == "edges":        # exactly on, just above and below the dyadic edges
        e = y1 * 2.0 ** -np.floor(np.log2(y1 / top) + 12 * g.random(M))
        y = e * (1 + np.array([0.0, 2.0 ** -40, -2.0 ** -40])[g.integers(0, 3, M)])
    else:                        # one band
        y = top * (0.26 + 0.2 * g.random(M))
    return np.stack([x, y / (2 * np.pi)], -1)


def _bound(prec, eps, ref, x):
    return eps if prec != "fp32" else eps + 32 * U32 * np.max(np.abs(ref)) / np.sum(np.abs(x))


@pytest.mark.parametrize("kind", ["octaves", "uniform", "edges", "single"])
@pytest.mark.parametrize("prec,eps,N,M", [("fp64", 1e-12, 5000, 4000), ("fp64", 1e-6, 4097, 3001),
                                          ("fp64ff", 1e-12, 5000, 4000), ("fp32", 1e-6, 270001, 60001),
                                          ("fp32", 1e-4, 300000, 20000)])
def test_merged_bands(fl, kind, prec, eps, N, M):
    dev = torch.device("cuda")
    cdt = torch.complex64 if prec == "fp32" else torch.complex128
    w = _nodes(kind, N, M, eps, seed=N + M)
    c, r = W.coefficients(N, seed=1), W.coefficients(M, seed=2)
    plan = fl.Plan(N, torch.from_numpy(w).to(dev), eps, precision=prec)
    ct, rt = torch.from_numpy(c).to(cdt).to(dev), torch.from_numpy(r).to(cdt).to(dev)
    f = plan.execute(ct).cpu().numpy().astype(np.complex128)
    d = plan.execute(ct, deriv=True).cpu().numpy().astype(np.complex128)
    g = plan.adjoint(rt).cpu().numpy().astype(np.complex128)
    plan.close()
    idx = np.sort(np.random.default_rng(3).choice(M, min(M, 400), replace=False))
    ref = oracle.flt_direct(c, w[idx])
    assert oracle.error_E(ref, f[idx], c) <= _bound(prec, eps, ref, c)
    cw = 2j * np.pi * np.arange(N) * c
    refd = oracle.flt_direct(cw, w[idx])
    assert oracle.error_E(refd, d[idx], cw) <= _bound(prec, eps, refd, cw)
    ks = np.sort(np.random.default_rng(4).choice(N, min(N, 400), replace=False))
    refa = oracle.flt_adjoint_at(r, w, ks)
    assert oracle.error_E(refa, g[ks], r) <= _bound(prec, eps, refa, r)
    nf = fl.Plan(N, torch.from_numpy(w).to(dev), eps, precision=prec, route="nfft")
    f0 = nf.execute(ct).cpu().numpy().astype(np.complex128)
    nf.close()
    assert oracle.error_E(f0, f, c) <= 2 * _bound(prec, eps, ref, c)


@pytest.mark.parametrize("kind", ["octaves", "single"])
@pytest.mark.parametrize("prec,eps", [("fp32", 1e-6), ("fp64", 1e-10)])
def test_merged_bands_real_exponents(fl, kind, prec, eps):
    N, M = 5000, 3000
    dev = torch.device("cuda")
    cdt = torch.complex64 if prec == "fp32" else torch.complex128
    w = _nodes(kind, N, M, eps, seed=9)
    w[:, 0] -= 0.5
    xi = np.random.default_rng(10).uniform(1.0, N, N)
    c, r = W.coefficients(N, seed=1), W.coefficients(M, seed=2)
    plan = fl.XiPlan(torch.from_numpy(xi).to(dev), torch.from_numpy(w).to(dev), eps, precision=prec)
    f = plan.execute(torch.from_numpy(c).to(cdt).to(dev)).cpu().numpy().astype(np.complex128)
    g = plan.transposed(torch.from_numpy(r).to(cdt).to(dev)).cpu().numpy().astype(np.complex128)
    plan.close()
    ref = oracle.xi_direct(c, xi, w[:300])
    assert oracle.error_E(ref, f[:300], c) <= _bound(prec, eps, ref, c)
    refg = oracle.xi_transposed(r, xi[:300], w)
    assert oracle.error_E(refg, g[:300], r) <= _bound(prec, eps, refg, r)


@pytest.mark.parametrize("prec,eps", [("fp32", 1e-6), ("fp64", 1e-10)])
def test_real_exponents_band_without_exponents(fl, prec, eps):
    # every exponent above the low bands' cuts: those bands' sums are empty
    N, M = 500, 400
    dev = torch.device("cuda")
    cdt = torch.complex64 if prec == "fp32" else torch.complex128
    w = W.nodes_disk_uniform(M, seed=11)
    w[:, 0] -= 0.5
    xi = np.random.default_rng(12).uniform(900.0, 1000.0, N)
    c, r = W.coefficients(N, seed=1), W.coefficients(M, seed=2)
    plan = fl.XiPlan(torch.from_numpy(xi).to(dev), torch.from_numpy(w).to(dev), eps, precision=prec)
    f = plan.execute(torch.from_numpy(c).to(cdt).to(dev)).cpu().numpy().astype(np.complex128)
    g = plan.transposed(torch.from_numpy(r).to(cdt).to(dev)).cpu().numpy().astype(np.complex128)
    plan.close()
    ref, refg = oracle.xi_direct(c, xi, w), oracle.xi_transposed(r, xi, w)
    assert oracle.error_E(ref, f, c) <= _bound(prec, eps, ref, c)
    assert oracle.error_E(refg, g, r) <= _bound(prec, eps, refg, r)
