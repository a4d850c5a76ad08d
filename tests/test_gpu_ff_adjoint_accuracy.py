"""The float-pair adjoint at N = M = 2^18, eps = 1e-12, in the relative 2-norm over
sampled frequencies.  Bar: pairs round at 2^-46 per operation (unnormalised sums
and products); the window's 24 taps, the 2 x 20 layers of the grids' FFTs and the
up to 130 terms of a frequency's sum over grids and right-hand sides add up as
independent roundings, times the deconvolution's gain of at most 8.6 at m_w = 8."""
import numpy as np
import pytest

import oracle
from paper_1606_03255_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
BAR = 8.6 * np.sqrt(24 + 40 + 130) * 2.0 ** -46


@pytest.fixture(scope="module")
def fl():
    from paper_1606_03255_gb300 import build as libbuild
    libbuild.build()
    from paper_1606_03255_gb300 import fl as flmod
    flmod.load()
    return flmod


@pytest.mark.parametrize("nodes", ["disk", "circle"])
def test_ff_adjoint(fl, nodes):
    N = M = 1 << 18
    w = W.nodes_disk_uniform(M, seed=1) if nodes == "disk" else W.nodes_circle_clustered(M, seed=1)
    r = W.coefficients(M, seed=2)
    dev = torch.device("cuda")
    plan = fl.Plan(N, torch.from_numpy(w).to(dev), 1e-12, precision="fp64ff")
    g = plan.adjoint(torch.from_numpy(r).to(dev)).cpu().numpy()
    plan.close()
    ks = np.sort(np.random.default_rng(3).choice(N, 256, replace=False))
    ref = oracle.flt_adjoint_at(r, w, ks)
    assert np.linalg.norm(g[ks] - ref) / np.linalg.norm(ref) <= BAR
