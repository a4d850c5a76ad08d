"""FP64 plans with merged bands err no more, against the oracle, than plans whose
bands are interpolated one by one (route "nfft", which merges none): product and
adjoint, relative 2-norms, above a floor of 64 units of rounding."""
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


def _rel(a, ref):
    return np.linalg.norm(a - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("eps", [1e-8, 1e-10, 1e-12])
@pytest.mark.parametrize("N,M", [(300, 5000), (2048, 4096), (3000, 3000), (4097, 2403)])
def test_merged_no_less_accurate(fl, N, M, eps):
    w = W.nodes_circle_clustered(M, seed=N)
    c, r = W.coefficients(N, seed=1), W.coefficients(M, seed=2)
    ref, refa = oracle.flt_direct(c, w), oracle.flt_adjoint(r, w, N)
    dev = torch.device("cuda")
    err = {}
    for route in ("auto", "nfft"):
        plan = fl.Plan(N, torch.from_numpy(w).to(dev), eps, precision="fp64", route=route)
        f = plan.execute(torch.from_numpy(c).to(dev)).cpu().numpy()
        g = plan.adjoint(torch.from_numpy(r).to(dev)).cpu().numpy()
        plan.close()
        err[route] = (_rel(f, ref), _rel(g, refa))
    for merged, single in zip(err["auto"], err["nfft"]):
        assert merged <= max(single, 64 * 2.0 ** -53), err
