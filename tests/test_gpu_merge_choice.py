"""Bands are merged where that is faster: on the sizes where merging directly summed
bands cost up to three times their direct sums, a default plan takes no longer than
1.15 times
the plan of the same rank given by the caller, which merges none."""
import numpy as np
import pytest

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


def _time(call):
    for _ in range(5):
        call()
    best = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            call()
        b.record()
        torch.cuda.synchronize()
        best.append(a.elapsed_time(b))
    return min(best)


@pytest.mark.parametrize("prec,eps,N,M", [("fp64", 1e-10, 1024, 1000), ("fp64", 1e-10, 65536, 1000),
                                          ("fp64ff", 1e-10, 256, 10000), ("fp64ff", 1e-10, 1024, 3000),
                                          ("fp32", 1e-6, 270001, 3000), ("fp32", 1e-6, 600000, 3000)])
def test_merging_does_not_slow_down(fl, prec, eps, N, M):
    dt = torch.complex64 if prec == "fp32" else torch.complex128
    dev = torch.device("cuda")
    w = torch.from_numpy(W.nodes_circle_clustered(M, seed=N)).to(dev)
    c = torch.from_numpy(W.coefficients(N, seed=1)).to(dt).to(dev)
    out = torch.empty(M, dtype=dt, device=dev)
    plan = fl.Plan(N, w, eps, precision=prec)
    plain = fl.Plan(N, w, eps, precision=prec, q=plan.info()["q"])
    ours, theirs = _time(lambda: plan.execute(c, out=out)), _time(lambda: plain.execute(c, out=out))
    plan.close()
    plain.close()
    assert ours <= 1.15 * theirs, (ours, theirs)
