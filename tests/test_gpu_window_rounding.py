"""The FP64 NFFT at eps = 1e-12 errs by rounding alone, and by less than its window's
argument would lose: b r of sinh reaches b m_w = 38, whose rounding by half a unit
moves a window value by 38 2^-53 = 4.2e-15.  The relative 2-norm error against the
oracle stays below half of that, for single plans (tables) and batches (windows
formed in the call), product and adjoint."""
import numpy as np
import pytest

import oracle
from paper_1606_03255_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
BAR = 0.5 * 38 * 2.0 ** -53


@pytest.fixture(scope="module")
def fl():
    from paper_1606_03255_gb300 import build as libbuild
    libbuild.build()
    from paper_1606_03255_gb300 import fl as flmod
    flmod.load()
    return flmod


@pytest.mark.parametrize("N,M", [(1000, 3000), (2048, 4096), (5000, 3000)])
def test_fp64_window_rounding(fl, N, M):
    w = W.nodes_circle_clustered(M, seed=N)
    w[:, 1] = 0.0                                          # one plain NFFT
    c, r = W.coefficients(N, seed=1), W.coefficients(M, seed=2)
    dev = torch.device("cuda")
    wt, ct, rt = (torch.from_numpy(x).to(dev) for x in (w, c, r))
    ref, refa = oracle.flt_direct(c, w), oracle.flt_adjoint(r, w, N)
    plan = fl.Plan(N, wt, 1e-12, precision="fp64", route="nfft")
    batch = fl.BatchedPlan([N], [M], wt, 1e-12, precision="fp64", route="nfft")
    for out, want in ((plan.execute(ct), ref), (batch.execute(ct), ref), (plan.adjoint(rt), refa)):
        err = np.linalg.norm(out.cpu().numpy() - want) / np.linalg.norm(want)
        assert err <= BAR, err
    plan.close()
    batch.close()
