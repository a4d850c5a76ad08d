"""Calls of one Laplace plan one after the other on a stream, each with other
coefficients written just before it, give the same bits as calls with a
synchronisation between them: the kernels of a call overlap their launches, and
none may read what an earlier call left in the plan's buffers.  Plans whose first
kernel is not the moments (no element, or one band) included."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fl():
    from paper_1606_03255_gb300 import build as libbuild
    libbuild.build()
    from paper_1606_03255_gb300 import fl as flmod
    flmod.load()
    return flmod


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kernel,N,M,t1", [("laplace", 1, 1, 1.0), ("laplace", 700, 5000, 1.0),
                                           ("laplace", 1 << 16, 300, 1.0), ("laplace", 0, 400, 1.0),
                                           ("exp", 5000, 700, 1.0), ("exp", 300, 400, 0.0),
                                           ("bessel_half", 3000, 3000, 1.0)])
def test_back_to_back_calls(fl, prec, kernel, N, M, t1):
    dev = torch.device("cuda")
    rdt = torch.float64 if prec == "fp64" else torch.float32
    rng = np.random.default_rng(N + M)
    t = torch.from_numpy(t1 * rng.uniform(1e-3, 1.0, N)).to(dev)     # t1 = 0: one band, no moments
    s = torch.from_numpy(rng.uniform(1e-3, 2.0 * max(N, 1), M)).to(dev)
    plan = fl.LaplacePlan(t, s, 1e-6, precision=prec, kernel=kernel)
    cs = torch.from_numpy(rng.standard_normal((24, N))).to(rdt).to(dev)
    c = torch.empty(N, dtype=rdt, device=dev)
    serial = []
    for x in cs:
        c.copy_(x)
        torch.cuda.synchronize()
        serial.append(plan.execute(c).clone())
        torch.cuda.synchronize()
    outs = [torch.empty(M, dtype=rdt, device=dev) for _ in cs]
    for _ in range(3):
        for x, o in zip(cs, outs):
            c.copy_(x)
            plan.execute(c, out=o)
        torch.cuda.synchronize()
        for a, b in zip(serial, outs):
            assert torch.equal(a, b)
    plan.close()
