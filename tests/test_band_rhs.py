"""The right-hand sides that a plan reports for its bands: what the grids' bytes are
counted from.  Bands evaluated together count once (planned on the stand-in for the
CUDA runtime, CPU), and the bench's method bytes follow the plan's numbers."""
import ctypes

import bench
from test_plan_resources import _data, _ptr, lib, vp  # noqa: F401  (lib: fixture)
from paper_1606_03255_gb300 import fl

import numpy as np


def test_merged_bands_count_once(lib):  # noqa: F811
    N = M = 300000
    nodes = np.zeros((M, 2))
    out = ctypes.c_void_p()
    cb = _data(M, 9)
    lib.fake_d2h(cb)
    lib.fake_reset(-1)
    assert lib.fl_plan(ctypes.byref(out), N, M, _ptr(nodes), 0, 1e-6, 0, None) == 0
    info = fl.fl_info()
    assert lib.fl_get_info(out, ctypes.byref(info)) == 0
    rhs = (ctypes.c_int * 128)()
    assert lib.fl_get_band_rhs(out, rhs, 128) == 0 and lib.fl_get_band_rhs(out, rhs, 129) != 0
    nfft = [b for b in range(1, info.levels + 1) if info.band_route[b] == 1]
    assert rhs[0] == 0 and rhs[info.levels] == 1 and not any(rhs[info.levels + 1:])
    assert sum(1 for b in nfft if rhs[b] == 0) > 0                 # some were merged into an earlier one
    assert sum(rhs) < info.q * (len(nfft) - 1) + 1
    d = fl.info_dict(info)
    counted = bench.method_bytes({**d, "band_rhs": list(rhs)[:info.levels + 1]}, info.q)
    assert counted == sum(rhs[b] * info.band_parts[b] * 16.0 * info.band_n[b] for b in nfft)
    assert counted < bench.method_bytes(d, info.q)
    lib.fl_destroy(out)
