"""The FP32 adjoint turns its result by no common angle: the centring and sub-band
phases are the floats nearest to their fractions, so that their errors average
out over the nodes.  Fractions cut off at 24 bits would turn every node by 2^-25
turns on average; the bar is half of that."""
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


@pytest.mark.parametrize("N", [1735, 3000, 40001])       # one grid; sub-bands at 40001
def test_no_common_turn(fl, N):
    M = 4000
    w = np.stack([np.random.default_rng(N).random(M), np.zeros(M)], axis=1)
    r = W.coefficients(M, seed=2).astype(np.complex64)
    plan = fl.Plan(N, torch.from_numpy(w).to("cuda"), 1e-7, precision="fp32", route="nfft")
    g = plan.adjoint(torch.from_numpy(r).to("cuda")).cpu().numpy().astype(np.complex128)
    plan.close()
    ref = oracle.flt_adjoint(r.astype(np.complex128), w, N)
    angle = np.angle(np.vdot(ref, g))
    assert abs(angle) <= 2 * np.pi * 2.0 ** -26, angle
