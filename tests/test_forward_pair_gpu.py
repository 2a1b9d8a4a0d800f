"""The FP32 passes of the grid-to-coefficients transform at all lengths they are
compiled for (64 .. 4096 in each direction) and just below, against the
oracle's doubled-torus sums: the fewest columns (blocks with one column in use),
odd numbers of fields, members, both parities, outputs that are 8-byte but not
16-byte aligned, and the half spectrum that real-field plans interpolate from.

Tolerance of the coefficients: 2e-6 of the largest (rounding of order 6e-8 times
log2(N1 N2) <= 18 levels, and a margin of two)."""
import numpy as np
import pytest

import oracle
from paper_2605_01313_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for the -m gpu tests")
    build.build()
    return torch


def plan_for(n_lon, n_lat, F, members=1, real=True):
    from paper_2605_01313_gb300 import Plan
    from paper_2605_01313_gb300.nufft import Options
    return Plan(n_lon, n_lat, 1e-6, "f32", F, n_members=members,
                options=Options.make(real_fields=real))


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("n_lon,n_lat,members", [(16, 16, 1), (16, 32, 3), (64, 64, 1),
                                                 (16, 128, 1), (16, 256, 2), (32, 512, 1),
                                                 (64, 512, 3), (16, 1024, 1), (64, 1024, 2),
                                                 (16, 2048, 1), (64, 8, 1),
                                                 (128, 16, 2), (256, 8, 1), (4096, 8, 1)])
def test_coefficients(torch_cuda, n_lon, n_lat, members, aligned):
    torch = torch_cuda
    rng = np.random.default_rng(n_lon + n_lat + members)
    F, par = 3, [-1, 1, -1]
    s = rng.standard_normal((members, F, n_lat, n_lon)).astype(np.float32)
    with plan_for(n_lon, n_lat, F, members) as plan:
        shape = plan.coeff_shape
        n = int(np.prod(shape))
        buf = torch.zeros(n + 2, dtype=torch.complex64, device="cuda")
        off = 0 if aligned else 1
        x = torch.from_numpy(s if members > 1 else s[0]).cuda()
        plan.grid_to_coeffs(x, par, out=buf[off:off + n].view(shape))
        plan.check()
        got = buf.cpu().numpy()
    assert not got[:off].any() and not got[off + n:].any()
    got = got[off:off + n].reshape((members, F, 2 * n_lat, n_lon))
    for k in range(members):
        ref = oracle.grid_to_coeffs(s[k].astype(np.float64), par)
        assert np.max(np.abs(got[k] - ref)) <= 2e-6 * np.max(np.abs(ref))


@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("n_lon,n_lat", [(16, 256), (32, 512), (16, 1024)])
def test_interpolation_from_the_grid(torch_cuda, n_lon, n_lat, real):
    torch = torch_cuda
    rng = np.random.default_rng(7 * n_lon + n_lat)
    par, P = [1, -1, 1], 157
    s = rng.standard_normal((3, n_lat, n_lon)).astype(np.float32)
    lon, colat = rng.uniform(-1.0, 7.0, P), rng.uniform(0.0, np.pi, P)
    with plan_for(n_lon, n_lat, 3, real=real) as plan:
        plan.set_points(torch.from_numpy(lon).cuda(), torch.from_numpy(colat).cuda())
        v = plan.interpolate_grid(torch.from_numpy(s).cuda(), par).cpu().numpy()
        plan.check()
    ref = oracle.evaluate(oracle.grid_to_coeffs(s.astype(np.float64), par), lon, colat)
    for f in range(3):
        assert oracle.rel_linf(v[f], ref[f].real) <= 2e-5
