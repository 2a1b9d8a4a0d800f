"""Device pointers off their element's size are refused on the host (reading them
would fault on the device): every entry point, both precisions.  Each call must
return before anything is launched; the plan then works as before."""
import ctypes

import numpy as np
import pytest

from paper_2605_01313_gb300 import build, nufft
from paper_2605_01313_gb300.nufft import Options

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for the -m gpu tests")
    build.build()
    return torch


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_misaligned_pointers_are_refused(torch_cuda, dtype):
    from paper_2605_01313_gb300 import Ensemble, Plan
    torch = torch_cuda
    real = 8 if dtype == "f64" else 4
    tol = 1e-12 if dtype == "f64" else 1e-6
    rd, cd = (torch.float64, torch.complex128) if dtype == "f64" else \
        (torch.float32, torch.complex64)
    n_lon, n_lat, P = 64, 32, 100
    lon = torch.linspace(0, 6, P, dtype=torch.float64, device="cuda")
    colat = torch.linspace(0.1, 3, P, dtype=torch.float64, device="cuda")
    room = torch.zeros(2 * 64 * 64 + 64, dtype=torch.float64, device="cuda").data_ptr()
    par = np.array([1], dtype=np.int32)
    L = nufft.lib()
    vp = ctypes.c_void_p
    bad = nufft.ERR_INVALID_ARG
    with Plan(n_lon, n_lat, tol, dtype, 1, options=Options.make(real_fields=True)) as plan:
        h = plan._h
        one = np.array([P], dtype=np.int64)
        pts = lon.data_ptr(), colat.data_ptr()
        assert L.dfsnufft_set_points_batch(h, one.ctypes.data, vp(pts[0] + 4), vp(pts[1])) == bad
        assert L.dfsnufft_set_points_batch(h, one.ctypes.data, vp(pts[0]), vp(pts[1] + 4)) == bad
        plan.set_points(lon, colat)
        for c, v in ((room + real, room), (room, room + real // 2)):
            assert L.dfsnufft_execute(h, vp(c), vp(v)) == bad
            assert L.dfsnufft_execute_pr(h, 10, 10, vp(c), vp(v)) == bad
            assert L.dfsnufft_grid_to_coeffs(h, vp(v), par.ctypes.data, vp(c)) == bad
            assert L.dfsnufft_execute_noalloc(n_lon, n_lat, tol, plan.params["dtype"], 1, P,
                                              vp(pts[0]), vp(pts[1]), vp(c), vp(v), None) == bad
        assert L.dfsnufft_execute_noalloc(n_lon, n_lat, tol, plan.params["dtype"], 1, P,
                                          vp(pts[0] + 4), vp(pts[1]), vp(room), vp(room),
                                          None) == bad
        for s, v in ((room + real // 2, room), (room, room + real // 2)):
            assert L.dfsnufft_interpolate_grid(h, vp(s), par.ctypes.data, vp(v)) == bad
        coeffs = torch.zeros((1, 2 * n_lat, n_lon), dtype=cd, device="cuda")
        coeffs[0, n_lat, n_lon // 2] = 3.0            # the constant 3
        vals = plan.execute(coeffs)
        plan.check()
        assert torch.allclose(vals, torch.full_like(vals, 3.0), rtol=1e-5)
    ens = Ensemble([(1, n_lon, n_lat)], tol=tol, dtype=dtype, n_fields=1)
    out = torch.empty(P, dtype=rd, device="cuda")
    arr = lambda x: (vp * 1)(x)
    good = [arr(one.ctypes.data), arr(pts[0]), arr(pts[1]), arr(coeffs.data_ptr()),
            arr(out.data_ptr())]
    for k, off in ((1, 4), (2, 4), (3, real), (4, real // 2)):
        args = list(good)
        args[k] = arr(good[k][0] + off)
        assert L.dfsnufft_ensemble_run(ens._h, *args) == bad
    assert L.dfsnufft_ensemble_run(ens._h, *good) == nufft.OK
    ens.check()
    assert torch.allclose(out, torch.full_like(out, 3.0), rtol=1e-5)
    ens.destroy()
