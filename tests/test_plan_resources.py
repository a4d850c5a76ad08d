"""What planning allocates, and that it gives everything back: the library's objects
linked with a stand-in for the CUDA runtime (fake_cudart.c) that counts device
allocations and fails the n-th one.  Every plan call, failed at each of its
allocations in turn, reports FL_ENOMEM and leaves nothing allocated; a plan that is
made holds few allocations and frees them all (CPU)."""
import ctypes
import glob
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FP32, FP64, FF = 0, 1, 2
vp, i64, ci, cd = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, ctypes.c_double


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("gcc") or not shutil.which("g++"):
        pytest.skip("no host compiler")
    from paper_1606_03255_gb300 import build as libbuild
    libbuild.build()
    d = tmp_path_factory.mktemp("fake")
    obj, so = str(d / "fake.o"), str(d / "libfl_fake.so")
    subprocess.run(["gcc", "-O1", "-fPIC", "-c", os.path.join(ROOT, "tests", "fake_cudart.c"), "-o", obj], check=True)
    objs = [os.path.join(libbuild.BUILD, os.path.basename(s)[:-3] + ".o")
            for s in sorted(glob.glob(os.path.join(libbuild.SRC, "*.cu")))]
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so, *objs, obj], check=True)
    h = ctypes.CDLL(so)
    h.fl_plan.argtypes = [vp, i64, i64, vp, ci, cd, ci, vp]
    h.fl_plan_xi.argtypes = [vp, i64, vp, i64, vp, ci, cd, ci, vp]
    h.fl_plan_laplace.argtypes = [vp, i64, i64, vp, vp, ci, cd, ci, vp]
    h.fl_plan_kernel.argtypes = [vp, ci, i64, i64, vp, vp, ci, cd, ci, vp]
    h.fl_plan_batched.argtypes = [vp, ci, vp, vp, vp, ci, cd, ci, vp, vp]
    h.fl_destroy.argtypes = [vp]
    h.fake_reset.argtypes = [ctypes.c_long]
    h.fake_live.restype = h.fake_made.restype = ctypes.c_long
    return h


CALLBACK = ctypes.CFUNCTYPE(None, vp, ctypes.c_size_t)


def _data(M, near):
    """Device-to-host data: two doubles are the ends of the Laplace intervals, longer
    arrays of 8-byte words band counts (the nodes spread evenly over some bands)."""
    def fill(dst, n):
        if n == 16:
            np.ctypeslib.as_array(ctypes.cast(dst, ctypes.POINTER(cd)), (2,))[:] = (1.0, 2000.0)
        elif n >= 64 and n % 8 == 0:
            a = np.ctypeslib.as_array(ctypes.cast(dst, ctypes.POINTER(i64)), (n // 8,))
            if not a.any():
                a[near:near + 12] = M // 13
                a[-1] = M - 12 * (M // 13)
    return CALLBACK(fill)


def _ptr(a):
    return a.ctypes.data_as(vp)


def _calls(h):
    """name -> plan call, on host arrays."""
    rng = np.random.default_rng(1)
    N = M = 3000
    nodes = np.stack([rng.random(M) - 0.5, rng.random(M)], 1)
    t, s, xi = rng.random(N), rng.random(M), 1.0 + rng.random(N) * N
    big = np.stack([rng.random(300000), rng.random(300000)], 1)
    Ns = np.array([500, 3000, 40], dtype=np.int64)
    keep = (nodes, t, s, xi, big, Ns)
    out = ctypes.c_void_p()
    o = ctypes.byref(out)
    calls = {"fp%d" % p: (lambda p=p: h.fl_plan(o, N, M, _ptr(nodes), 0, 1e-10, p, None)) for p in (FP64, FF)}
    calls["fp32 270000"] = lambda: h.fl_plan(o, 270000, 300000, _ptr(big), 0, 1e-6, FP32, None)
    calls["fp32"] = lambda: h.fl_plan(o, N, M, _ptr(nodes), 0, 1e-6, FP32, None)
    calls["xi"] = lambda: h.fl_plan_xi(o, N, _ptr(xi), M, _ptr(nodes), 0, 1e-6, FP32, None)
    calls["batched"] = lambda: h.fl_plan_batched(o, 3, _ptr(Ns), _ptr(Ns), _ptr(big), 0, 1e-6, FP32, None, None)
    calls["laplace"] = lambda: h.fl_plan_laplace(o, N, M, _ptr(t), _ptr(s), 0, 1e-6, FP64, None)
    calls["exp"] = lambda: h.fl_plan_kernel(o, 1, N, M, _ptr(t), _ptr(s), 0, 1e-6, FP64, None)
    calls["bessel_half"] = lambda: h.fl_plan_kernel(o, 2, N, M, _ptr(t), _ptr(s), 0, 1e-6, FP32, None)
    return calls, out, keep


NAMES = ["fp1", "fp2", "fp32", "fp32 270000", "xi", "batched", "laplace", "exp", "bessel_half"]


@pytest.mark.parametrize("near", [2, 9])
@pytest.mark.parametrize("name", NAMES)
def test_failed_plans_leave_nothing(lib, name, near):
    calls, out, keep = _calls(lib)
    cb = _data(300000 if "270000" in name else 500 if name == "batched" else 3000, near)
    lib.fake_d2h(cb)
    lib.fake_reset(-1)
    assert calls[name]() == 0
    made = lib.fake_made()
    lib.fl_destroy(out)
    assert lib.fake_live() == 0
    for k in range(made):
        lib.fake_reset(k)
        assert calls[name]() == 2, k                       # FL_ENOMEM
        assert lib.fake_live() == 0, k


@pytest.mark.parametrize("name", ["fp1", "fp2", "fp32", "laplace"])
def test_small_plans_make_few_allocations(lib, name):
    # each costs microseconds, and small tables share blocks
    calls, out, keep = _calls(lib)
    cb = _data(3000, 9)
    lib.fake_d2h(cb)
    lib.fake_reset(-1)
    assert calls[name]() == 0
    assert lib.fake_made() <= 12
    lib.fl_destroy(out)
