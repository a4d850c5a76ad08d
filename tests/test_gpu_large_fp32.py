"""FP32 transforms of more than 2^18 coefficients, whose forward steps are free to
round as they like: direct sums with z and z^8 from plan time and several blocks
per lane (node pairs with an odd one, frequency counts on both sides of a block
and of a chunk, powers from one to underflow within a pair), and default plans,
whose gathers are fused or not by cost.  Against the oracle with the bounds of
the forward, gradient and adjoint tests."""
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


def _bound(eps, ref, x):
    return eps + 32 * U32 * np.max(np.abs(ref)) / np.sum(np.abs(x))


# bands keep 2^j + 1 frequencies at N = 2^18 + 1, 2^j at 2^19
@pytest.mark.parametrize("N", [(1 << 18) + 1, 1 << 19])
@pytest.mark.parametrize("M", [1, 2, 33, 515])
def test_direct_items(fl, N, M):
    dev, eps = torch.device("cuda"), 1e-6
    rng = np.random.default_rng(N + M)
    y = 10.0 ** rng.uniform(-9.0, np.log10(np.log(1.0 / eps)), M)
    w = np.stack([rng.random(M), y / (2 * np.pi)], axis=1)
    w[::5, 1] = 0.0
    c, r = W.coefficients(N, seed=1), W.coefficients(M, seed=2)
    plan = fl.Plan(N, torch.from_numpy(w).to(dev), eps, precision="fp32", route="direct")
    assert plan.info()["n_bands_fft"] == 0
    ct, rt = (torch.from_numpy(x).to(torch.complex64).to(dev) for x in (c, r))
    f, g, gw = (x.cpu().numpy().astype(np.complex128) for x in (plan.execute(ct), plan.adjoint(rt), plan.grad_w(ct, rt)))
    plan.close()
    ref = oracle.flt_direct(c, w)
    assert oracle.error_E(ref, f, c) <= _bound(eps, ref, c)
    ks = np.unique(np.concatenate([np.arange(70), np.arange(500, 530), np.arange(4080, 4110), rng.integers(0, N, 200)]))
    refa = oracle.flt_adjoint_at(r, w, ks)
    assert oracle.error_E(refa, g[ks], r) <= _bound(eps, refa, r)
    cw = 2j * np.pi * np.arange(N) * c
    refd = oracle.flt_direct(cw, w)
    err = np.max(np.abs(gw - r * np.conj(refd)))
    assert err <= eps * np.max(np.abs(r)) * np.sum(np.abs(cw)) + 32 * U32 * np.max(np.abs(r * refd))


@pytest.mark.parametrize("fuse", ["auto", "on", "off"])
@pytest.mark.parametrize("where", ["spread", "one cell", "ends"])
@pytest.mark.parametrize("M", [1, 1023, 1025, 40000])
def test_default_plans(fl, M, where, fuse):
    dev, N, eps = torch.device("cuda"), 300000, 1e-6
    rng = np.random.default_rng(M)
    x = rng.random(M)
    if where == "one cell":
        x = 0.37 + 1e-8 * x
    elif where == "ends":
        x = np.where(x < 0.5, 2e-5 * x, 1.0 - 2e-5 * (1.0 - x))
    w = np.stack([x, 10.0 ** (-6.0 * rng.random(M)) / (2 * np.pi)], axis=1)
    w[::2, 1] = 0.0
    c = W.coefficients(N, seed=M + 1)
    plan = fl.Plan(N, torch.from_numpy(w).to(dev), eps, precision="fp32", fuse=fuse)
    f = plan.execute(torch.from_numpy(c).to(torch.complex64).to(dev)).cpu().numpy().astype(np.complex128)
    plan.close()
    idx = np.sort(rng.choice(M, min(M, 300), replace=False))
    ref = oracle.flt_direct(c, w[idx])
    assert oracle.error_E(ref, f[idx], c) <= _bound(eps, ref, c)
