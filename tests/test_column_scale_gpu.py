"""Columns of small coefficients in FP64 plans: the theta pass carries each column
at its own power of two and the phi pass joins them, so a column must come through
at full accuracy whatever the others hold, down to subnormal numbers.

Reference: the FP64 oracle on the coefficients times 2^k, a power of two that
makes them normal numbers (exact, also for subnormal ones); the values times 2^k
are exact too.  Tolerance: 10 x the requested accuracy of the largest value, as
in every FP64 test (1e-11 at 1e-12)."""
import math

import numpy as np
import pytest

import oracle
from paper_2605_01313_gb300 import build
from test_fft_pair_gpu import mirror_substituted

pytestmark = pytest.mark.gpu

@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for the -m gpu tests")
    build.build()
    return torch


def check(torch, c, real, k=0, tol=1e-12):
    """Every field of c against the oracle, both times 2^k."""
    from paper_2605_01313_gb300 import Plan
    from paper_2605_01313_gb300.nufft import Options
    rng = np.random.default_rng(5)
    F, N2, N1 = c.shape
    lon, colat = rng.uniform(-1.0, 7.0, 150), rng.uniform(0.0, math.pi, 150)
    with Plan(N1, N2 // 2, tol, "f64", F, options=Options.make(real_fields=real)) as plan:
        plan.set_points(torch.from_numpy(lon).cuda(), torch.from_numpy(colat).cuda())
        vals = plan.execute(torch.from_numpy(c).cuda())
        plan.check()
        vals = np.ldexp(vals.cpu().numpy(), k)
    up = np.ldexp(c.real, k) + 1j * np.ldexp(c.imag, k)
    ref = oracle.evaluate(mirror_substituted(up) if real else up, lon, colat)
    for f in range(F):
        assert oracle.rel_linf(vals[f], ref[f].real) <= 10 * tol, f


def noise(rng, F, n_lon, n_lat):
    shape = (F, 2 * n_lat, n_lon)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


# amplitudes (1 + |m|)^-3 at scales where the columns from about |m| = 4, 10 and 20 on
# hold subnormal numbers only, and where all of them do
@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("scale", [1e-306, 1e-305, 1e-304, 1e-309])
@pytest.mark.parametrize("n_lon,n_lat", [(64, 32), (128, 20)])
def test_subnormal_columns(torch_cuda, n_lon, n_lat, scale, real):
    rng = np.random.default_rng(81)
    m = np.abs(np.arange(n_lon) - n_lon // 2)
    c = noise(rng, 2, n_lon, n_lat) * (scale * (1.0 + m) ** -3.0)
    assert (np.abs(c).max(axis=1) < np.finfo(float).tiny).any()
    check(torch_cuda, c, real, 1000)


# factors over what the bound resolves, and a smooth decay
@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("kind", ["random", "decay"])
def test_column_factors(torch_cuda, kind, real):
    rng = np.random.default_rng(82)
    c = noise(rng, 3, 80, 24)
    m = np.abs(np.arange(80) - 40)
    c *= 2.0 ** rng.uniform(-30, 0, (3, 1, 80)) if kind == "random" else (1.0 + m) ** -3.0
    check(torch_cuda, c, real)


# a field for each array column, which alone is large (by 2^20, and by 10^250): the
# line's scale is that column's, wherever its exponent is read
@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("factor", [2.0 ** -20, 1e-250])
def test_largest_column_anywhere(torch_cuda, factor, real):
    rng = np.random.default_rng(83)
    n_lon = 64
    c = noise(rng, n_lon, n_lon, 8) * factor
    for q in range(n_lon):
        c[q, :, q] /= factor
        if real and 0 < q < n_lon // 2:  # the column a real-field plan reads in its place
            c[q, :, n_lon - q] /= factor
    check(torch_cuda, c, real)


# the same at narrow rows and kernels, where the phi pass runs CTAs of less than a warp
@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("n_lon", [4, 6, 8])
def test_largest_column_in_part_warps(torch_cuda, n_lon, real):
    rng = np.random.default_rng(84)
    c = noise(rng, n_lon, n_lon, 16) * 2.0 ** -20
    for q in range(n_lon):
        c[q, :, q] *= 2.0 ** 20
        if real and 0 < q < n_lon // 2:
            c[q, :, n_lon - q] *= 2.0 ** 20
    check(torch_cuda, c, real, tol=1e-4)
