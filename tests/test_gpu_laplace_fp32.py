"""The FP32 form of planned Laplace transforms: no less accurate than its single
rounding of the result and the barycentric form of the allocation-free call allow
(relative 2-norms against the oracle at an eps where interpolation errs far
less than float rounding), and infinite coefficients leave the results that do
not depend on them finite and the others as the allocation-free call has them."""
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


def _both(fl, c, t, s, eps, prec="fp32"):
    """(planned, allocation-free) results."""
    dev = torch.device("cuda")
    rdt = torch.float32 if prec == "fp32" else torch.float64
    tt, ss, ct = (torch.from_numpy(np.asarray(x)).to(dev) for x in (t, s, c))
    ct = ct.to(rdt)
    plan = fl.LaplacePlan(tt, ss, eps, precision=prec)
    a = plan.execute(ct).cpu().numpy().astype(np.float64)
    plan.close()
    f = torch.zeros(len(s), dtype=rdt, device=dev)
    st = fl.fl_laplace_real_noalloc(len(t), len(s), tt.data_ptr(), ss.data_ptr(), ct.data_ptr(), f.data_ptr(), 0, eps,
                                    fl._precision(prec), torch.cuda.current_stream().cuda_stream)
    fl.check(st, "noalloc")
    return a, f.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("N,M", [(300, 5000), (1810, 8274), (2208, 4045), (20000, 5000), (200000, 3000)])
def test_fp32_rounding(fl, N, M):
    c, t, s = W.laplace_inputs(N, M, seed=N)
    c = c.astype(np.float32).astype(np.float64)
    ref = oracle.laplace_direct(c, t, s)
    a, b = _both(fl, c, t, s, 1e-9)
    ea, eb = (np.linalg.norm(x - ref) / np.linalg.norm(ref) for x in (a, b))
    assert ea <= max(eb, 2.0 ** -25), (ea, eb)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("value", [np.inf, -np.inf])
def test_infinite_coefficient(fl, prec, value):
    # t over 40 octaves, the infinite term at the smallest: the s_j with s t ~ 0 get an
    # infinity from the cumulative sum, the others (few) interpolate it
    rng = np.random.default_rng(3)
    N = M = 3000
    t = 2.0 ** -(40 * rng.random(N))
    s = 2.0 ** (30 * rng.random(M))
    c = rng.standard_normal(N).astype(np.float32).astype(np.float64)
    for k in (np.argmin(t), np.argmax(t)):
        d = c.copy()
        d[k] = value
        a, b = _both(fl, d, t, s, 1e-6, prec)
        assert np.array_equal(np.isfinite(a), np.isfinite(b))
        assert np.array_equal(a[np.isinf(b)], b[np.isinf(b)])
        both = np.isfinite(b)
        assert np.max(np.abs(a[both] - b[both]), initial=0.0) <= 1e-4 * np.sum(np.abs(c))
