"""GPU parity of the fused gather's plan-time entries at the edges of their chunks.

The entries of a fused band are made by one CTA per 1024 nodes; node counts on
both sides of that, all nodes in one grid cell, and windows across the grid's
end are checked against the FP64 oracle at E <= eps + 32 u_32 ||f||_inf / ||c||_1,
and two plans of the same nodes give the same bits (an entry's place does not
enter the sums).
"""
import numpy as np
import pytest

import oracle
from paper_1606_03255_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fl():
    from paper_1606_03255_gb300 import build as libbuild
    libbuild.build()
    from paper_1606_03255_gb300 import fl as flmod
    flmod.load()
    return flmod


@pytest.mark.parametrize("where", ["spread", "one cell", "ends"])
@pytest.mark.parametrize("M", [1, 1023, 1024, 1025, 2049])
def test_fused_entries(fl, M, where):
    N, eps = 40001, 1e-6
    rng = np.random.default_rng(M)
    x = rng.random(M)
    if where == "one cell":
        x = 0.37 + 1e-7 * x
    elif where == "ends":
        x = np.where(x < 0.5, 2e-4 * x, 1.0 - 2e-4 * (1.0 - x))
    w = np.stack([x, 10.0 ** (-6.0 * rng.random(M)) / (2 * np.pi)], axis=1)
    w[::2, 1] = 0.0
    c = W.coefficients(N, seed=M + 1)
    dev = torch.device("cuda")
    ct = torch.from_numpy(c).to(torch.complex64).to(dev)
    out = []
    for _ in range(2):
        plan = fl.Plan(N, torch.from_numpy(w).to(dev), eps, precision="fp32", route="nfft", fuse="on")
        out.append(plan.execute(ct).cpu().numpy())
        plan.close()
    assert np.array_equal(out[0], out[1])
    ref = oracle.flt_direct(c, w)
    tol = eps + 32 * 2.0 ** -24 * np.max(np.abs(ref)) / np.sum(np.abs(c))
    assert oracle.error_E(ref, out[0].astype(np.complex128), c) <= tol
