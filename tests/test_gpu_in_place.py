"""Results written over the coefficients (out = c, or overlapping it): the same bits
as with a result of its own, for plans whose bands are summed directly, by NFFTs or
both, with nodes in Z^0, in the three precisions, single (plain and replayed),
batched, derivative and node gradient."""
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


def _nodes(N, seed):
    w = W.nodes_disk_uniform(N, seed=seed)
    w[::7, 1] = 40.0                                       # Z^0
    return torch.from_numpy(w).to("cuda")


@pytest.mark.parametrize("prec,eps", [("fp32", 1e-6), ("fp64", 1e-10), ("fp64ff", 1e-10)])
@pytest.mark.parametrize("route", ["auto", "direct", "nfft"])
@pytest.mark.parametrize("N", [700, 40000])
def test_out_over_c(fl, prec, eps, route, N):
    dt = torch.complex64 if prec == "fp32" else torch.complex128
    c = torch.from_numpy(W.coefficients(N, seed=1)).to(dt).to("cuda")
    r = torch.from_numpy(W.coefficients(N, seed=2)).to(dt).to("cuda")
    for graph in (False, True):
        plan = fl.Plan(N, _nodes(N, 3), eps, precision=prec, route=route, use_graph=graph)
        with torch.cuda.stream(torch.cuda.Stream()):
            for call in (lambda x, o: plan.execute(x, out=o), lambda x, o: plan.execute(x, out=o, deriv=True),
                         lambda x, o: plan.grad_w(x, r, out=o)):
                ref = call(c, None)
                for shift in (0, 5):                       # out starts `shift` elements into c
                    buf = torch.zeros(N + shift, dtype=dt, device="cuda")
                    buf[:N] = c
                    assert torch.equal(call(buf[:N], buf[shift:]), ref)
            torch.cuda.synchronize()
        plan.close()


def test_out_over_c_batched(fl):
    Ns = [700, 5000, 1, 9000]
    w = torch.cat([_nodes(n, i) for i, n in enumerate(Ns)])
    c = torch.from_numpy(W.coefficients(sum(Ns), seed=4)).to(torch.complex64).to("cuda")
    plan = fl.BatchedPlan(Ns, Ns, w, 1e-6)
    with torch.cuda.stream(torch.cuda.Stream()):
        ref = plan.execute(c)
        for _ in range(2):
            x = c.clone()
            assert torch.equal(plan.execute(x, out=x), ref)
            assert torch.equal(plan.execute(c), ref)       # the replayed form as before
        torch.cuda.synchronize()
    plan.close()
