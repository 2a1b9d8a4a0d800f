"""The packed FP32 theta and phi passes at every length they are compiled for
(fine sizes 2^7 .. 2^13 in each direction) and just outside, against the FP64
oracle: real-field and general plans, white-noise coefficients with the Nyquist
row and column non-zero, columns that do not fill a block, ragged point counts.

Tolerance: 2e-5, the FP32 bound of every other test (20 x the requested
accuracy; rounding of the transforms adds a few 1e-7)."""
import math

import numpy as np
import pytest

import oracle
from paper_2605_01313_gb300 import build

pytestmark = pytest.mark.gpu

TOL_F32 = 2e-5


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for the -m gpu tests")
    build.build()
    return torch


def mirror_substituted(c):
    """What a real-field plan evaluates: off the Nyquist row, the columns
    -N1/2 < m < 0 are the conjugate mirrors of the columns -m."""
    F, N2, N1 = c.shape
    out = c.copy()
    q = np.arange(1, N1 // 2)
    out[:, 1:, q] = np.conj(c[:, :0:-1, :][:, :, N1 - q])
    return out


# (n_lon, n_lat): fine columns of 64 .. 8192 rows with few modes in longitude,
# then fine rows of 64 .. 8192 cells with few modes in latitude; n_lon = 22 is
# not a multiple of 4 (a real-field plan's columns then miss the TMA alignment)
GRIDS = [(12, 7), (12, 16), (20, 21), (44, 64), (12, 100), (36, 256), (12, 500), (20, 1024),
         (12, 1800), (22, 64), (64, 4), (76, 9), (200, 6), (512, 5), (520, 4), (1900, 4),
         (3000, 3)]


@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("n_lon,n_lat", GRIDS)
def test_every_length(torch_cuda, n_lon, n_lat, real):
    from paper_2605_01313_gb300 import Plan
    from paper_2605_01313_gb300.nufft import Options
    torch = torch_cuda
    rng = np.random.default_rng(1000 * n_lon + n_lat)
    F, N2, N1, P = 3, 2 * n_lat, n_lon, 301
    c = (rng.standard_normal((F, N2, N1)) + 1j * rng.standard_normal((F, N2, N1)))
    c = c.astype(np.complex64).astype(np.complex128)
    lon = rng.uniform(-1.0, 7.0, P)
    colat = rng.uniform(0.0, math.pi, P)
    with Plan(n_lon, n_lat, 1e-6, "f32", F, options=Options.make(real_fields=real)) as plan:
        plan.set_points(torch.from_numpy(lon).cuda(), torch.from_numpy(colat).cuda())
        out = plan.execute(torch.from_numpy(c).to(torch.complex64).cuda())
        plan.check()
        vals = out.cpu().numpy()
    ref = oracle.evaluate(mirror_substituted(c) if real else c, lon, colat)
    for f in range(F):
        assert oracle.rel_linf(vals[f], ref[f].real) <= TOL_F32
