"""A bin scan whose wait runs out (a chunk that never publishes its totals): the
timeout is reported, nothing downstream reads the unfinished bin list or the
records with gaps (the values are NaN and nothing outside them is written), and
the next set_points works."""
import math

import numpy as np
import pytest

import oracle
from paper_2605_01313_gb300 import build, nufft
from paper_2605_01313_gb300.nufft import Options

pytestmark = pytest.mark.gpu

CYCLES = 20_000_000                      # about 10 ms a chunk


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for the -m gpu tests")
    build.build()
    return torch


# the interpolation kernels: TMA boxes (w = 7), the general one (w = 9), fixed point
# (FP64); 2048 and more bins in 4 and more chunks, one member and three
@pytest.mark.parametrize("dtype,w,members", [("f32", 7, 1), ("f32", 9, 1), ("f32", 7, 3),
                                             ("f64", 0, 1), ("f64", 0, 3)])
def test_timed_out_scan_leaves_nothing_to_read(torch_cuda, dtype, w, members):
    from paper_2605_01313_gb300 import Plan
    torch = torch_cuda
    rng = np.random.default_rng(91)
    n_lon, n_lat, F, guard = 512, 256, 2, 4096
    counts = [30000, 5001, 77][:members]
    P = sum(counts)
    tile = (32, 16)
    lon, colat = rng.uniform(0, 2 * math.pi, P), rng.uniform(0, math.pi, P)
    lon_t, colat_t = torch.from_numpy(lon).cuda(), torch.from_numpy(colat).cuda()
    rd, cd = (torch.float64, torch.complex128) if dtype == "f64" else \
        (torch.float32, torch.complex64)
    k = 8                                # modes of the oracle's array
    small = rng.standard_normal((F, 2 * k, 2 * k)) + 1j * rng.standard_normal((F, 2 * k, 2 * k))
    small = small.astype(np.complex64).astype(np.complex128)
    small[:, 0, :] = small[:, :, 0] = 0.0
    c = np.zeros((F, 2 * n_lat, n_lon), dtype=np.complex128)
    c[:, n_lat - k:n_lat + k, n_lon // 2 - k:n_lon // 2 + k] = small
    c = torch.from_numpy(c).to(cd).cuda()
    if members > 1:
        c = c.expand(members, *c.shape).contiguous()
    buf = torch.full((F * P + 2 * guard,), 7.0, dtype=rd, device="cuda")
    vals = buf[guard:guard + F * P]
    with Plan(n_lon, n_lat, 1e-12 if dtype == "f64" else 1e-6, dtype, F, n_members=members,
              options=Options.make(w=w, tile=tile)) as plan:
        rc = nufft.dfsnufft_plan_selftest_scan_timeout(plan._h, counts, lon_t.data_ptr(),
                                                       colat_t.data_ptr(), CYCLES)
        assert rc == nufft.ERR_TIMEOUT
        assert nufft.dfsnufft_plan_point_stats(plan._h) == {"rows_needed": 0, "nonempty_bins": 0}
        nufft.dfsnufft_execute(plan._h, c.data_ptr(), vals.data_ptr())
        plan.check()
        assert torch.isnan(vals).all()
        assert (buf[:guard] == 7.0).all() and (buf[guard + F * P:] == 7.0).all()
        # the plan goes on
        plan.set_points(lon_t, colat_t, counts)
        vals.copy_(plan.execute(c).reshape(-1))
        plan.check()
    got = vals.cpu().numpy()
    for m, n in enumerate(counts):
        o = sum(counts[:m])
        v = got[F * o:F * (o + n)].reshape(F, n)[:, :300]
        ref = oracle.evaluate(small, lon[o:o + n][:300], colat[o:o + n][:300])
        for f in range(F):
            assert oracle.rel_linf(v[f], ref[f].real) <= (1e-11 if dtype == "f64" else 2e-5)


def test_selftest_refuses_plans_without_the_scan(torch_cuda):
    from paper_2605_01313_gb300 import Plan
    torch = torch_cuda
    x = torch.zeros(8, dtype=torch.float64, device="cuda")
    for n_lon, opts, cycles, code in ((64, Options.make(), CYCLES, nufft.ERR_UNSUPPORTED),
                                      (512, Options.make(keep_order=True), CYCLES,
                                       nufft.ERR_UNSUPPORTED),
                                      (512, Options.make(), 0, nufft.ERR_INVALID_ARG),
                                      (512, Options.make(), 5_000_000_000,
                                       nufft.ERR_INVALID_ARG)):
        with Plan(n_lon, n_lon // 2, 1e-6, "f32", 1, options=opts) as plan:
            assert nufft.dfsnufft_plan_selftest_scan_timeout(
                plan._h, [8], x.data_ptr(), x.data_ptr(), cycles) == code
            plan.check()
