"""Direct bands at the edges of their work items: the lanes per node (1 .. 32 as
K grows from one Horner block to a whole chunk), pairs of nodes with an odd one
left over, several chunks, segments made of neighbouring bands, and powers that
underflow; forward, node gradient and adjoint in the three arithmetics against
the oracle with the bounds of the forward and adjoint tests."""
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


def _bound(prec, eps, ref, x):
    return eps if prec != "fp32" else eps + 32 * U32 * np.max(np.abs(ref)) / np.sum(np.abs(x))


@pytest.mark.parametrize("prec,eps", [("fp32", 1e-6), ("fp64", 1e-12), ("fp64ff", 1e-12)])
@pytest.mark.parametrize("M", [1, 2, 33, 515])
@pytest.mark.parametrize("N", [1, 31, 32, 33, 65, 512, 513, 4096, 4097, 9000])
def test_direct_items(fl, prec, eps, N, M):
    dev = torch.device("cuda")
    cdt = torch.complex64 if prec == "fp32" else torch.complex128
    w = W.nodes_disk_uniform(M, seed=N + M)
    w[::3] = W.nodes_circle_clustered(M, seed=M)[::3]      # powers from 1 to underflow
    c, r = W.coefficients(N, seed=1), W.coefficients(M, seed=2)
    plan = fl.Plan(N, torch.from_numpy(w).to(dev), eps, precision=prec, route="direct")
    assert plan.info()["n_bands_fft"] == 0
    ct, rt = torch.from_numpy(c).to(cdt).to(dev), torch.from_numpy(r).to(cdt).to(dev)
    f = plan.execute(ct).cpu().numpy().astype(np.complex128)
    g = plan.adjoint(rt).cpu().numpy().astype(np.complex128)
    gw = plan.grad_w(ct, rt).cpu().numpy().astype(np.complex128)
    plan.close()
    ref = oracle.flt_direct(c, w)
    assert oracle.error_E(ref, f, c) <= _bound(prec, eps, ref, c)
    refa = oracle.flt_adjoint(r, w, N)
    assert oracle.error_E(refa, g, r) <= _bound(prec, eps, refa, r)
    cw = 2j * np.pi * np.arange(N) * c
    refd = oracle.flt_direct(cw, w)
    scale = np.max(np.abs(r)) * max(np.sum(np.abs(cw)), 1e-300)
    err = np.max(np.abs(gw - r * np.conj(refd)))
    rnd = 32 * U32 * np.max(np.abs(r * refd)) if prec == "fp32" else 0.0
    assert err <= eps * scale + rnd
