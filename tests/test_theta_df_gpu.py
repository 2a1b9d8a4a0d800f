"""The double-single theta pass of FP64 plans at every length it is compiled for
(2^6 .. 2^12 fine rows) and just outside, and its per-column scaling: columns of
magnitudes 400 orders apart, columns of zeros and of subnormal numbers, the
largest value in the Nyquist row or column; against the FP64 oracle.

Tolerance: 1e-11 of the largest value, the bound of every FP64 test at 1e-12."""
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


def check(torch, c, real, seed, bound=1e-11):
    from paper_2605_01313_gb300 import Plan
    from paper_2605_01313_gb300.nufft import Options
    rng = np.random.default_rng(seed)
    F, N2, N1 = c.shape
    lon, colat = rng.uniform(-1.0, 7.0, 211), rng.uniform(0.0, math.pi, 211)
    with Plan(N1, N2 // 2, 1e-12, "f64", F, options=Options.make(real_fields=real)) as plan:
        plan.set_points(torch.from_numpy(lon).cuda(), torch.from_numpy(colat).cuda())
        vals = plan.execute(torch.from_numpy(c).cuda())
        plan.check()
        vals = vals.cpu().numpy()
    ref = oracle.evaluate(mirror_substituted(c) if real else c, lon, colat)
    for f in range(F):
        assert oracle.rel_linf(vals[f], ref[f].real) <= bound


def noise(rng, F, n_lon, n_lat):
    shape = (F, 2 * n_lat, n_lon)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("n_lon,n_lat", [(12, 7), (12, 16), (22, 20), (44, 32), (12, 50),
                                         (36, 128), (12, 250), (20, 512), (12, 900), (8, 1024),
                                         (6, 1500)])
def test_every_length(torch_cuda, n_lon, n_lat, real):
    rng = np.random.default_rng(7 * n_lon + n_lat)
    check(torch_cuda, noise(rng, 2, n_lon, n_lat), real, n_lat)


@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("kind", ["spread", "zeros", "subnormal", "nyquist_row", "nyquist_col"])
def test_column_scales(torch_cuda, kind, real):
    rng = np.random.default_rng(71)
    c = noise(rng, 3, 48, 24)
    if kind == "spread":
        c *= 10.0 ** rng.uniform(-250, 150, (3, 1, 48))
    elif kind == "zeros":
        c[0, :, ::2] = 0.0
        c[1] = 0.0
        c[1, 30, 26] = 1.0
    elif kind == "subnormal":
        c[0, :, 20:40] *= 1e-310
        c[1] *= 1e-160
        c[1, :, 30:] *= 1e-155
    elif kind == "nyquist_row":
        c[:, 0, :] *= 1e60
    else:
        c[:, :, 0] *= 1e60
    check(torch_cuda, c, real, 72)
