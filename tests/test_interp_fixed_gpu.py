"""The FP64 plans' fixed-point interpolation at every kernel width and at the
magnitudes where its scaling can go wrong, against the FP64 oracle: tiny and
huge fields, fields of very different magnitude side by side, a field of zeros,
one that decays by 300 orders of magnitude, non-finite coefficients, points that
cannot be folded, one to five fields (one or two staging passes) and bins larger
than the grid.

Tolerance: ten times the requested accuracy, the bound of every other FP64 test
(1e-11 at 1e-12); the quantisation of tile values (2^-60 of the tile's largest)
and weights (2^-52) adds about 2e-16 of it."""
import math

import numpy as np
import pytest

import oracle
from paper_2605_01313_gb300 import build, synth

pytestmark = pytest.mark.gpu

# a tolerance whose width rule gives each width, 2 .. 16
TOL_OF_W = {2: 0.1, 3: 2e-2, 4: 3e-3, 5: 3e-4, 6: 3e-5, 7: 2e-6, 8: 4e-7, 9: 4e-8, 10: 4e-9,
            11: 5e-10, 12: 5e-11, 13: 4e-12, 14: 1e-12, 15: 1e-13, 16: 2e-14}


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for the -m gpu tests")
    build.build()
    return torch


def values(torch, c, lon, colat, n_lon, n_lat, tol=1e-12, **kw):
    from paper_2605_01313_gb300 import Plan
    from paper_2605_01313_gb300.nufft import Options
    with Plan(n_lon, n_lat, tol, "f64", c.shape[0], options=Options.make(**kw)) as plan:
        plan.set_points(torch.from_numpy(lon).cuda(), torch.from_numpy(colat).cuda())
        out = plan.execute(torch.from_numpy(c).cuda())
        plan.check()
        return out.cpu().numpy(), plan.params


def points(rng, n):
    return rng.uniform(0, 2 * math.pi, n), np.arccos(rng.uniform(-1, 1, n))


@pytest.mark.parametrize("w", sorted(TOL_OF_W))
def test_every_width(torch_cuda, w):
    rng = np.random.default_rng(w)
    wl = synth.small_workload(500 + w, 44, 22, n_fields=3, dtype="f64", points="uniform")
    lon, colat = points(rng, 1500)
    tol = TOL_OF_W[w]
    vals, prm = values(torch_cuda, wl.coeffs, lon, colat, 44, 22, tol)
    assert prm["w"] == w
    ref = oracle.evaluate(wl.coeffs, lon, colat)
    for f in range(3):
        assert oracle.rel_linf(vals[f], ref[f].real) <= 10 * tol


@pytest.mark.parametrize("n_fields", [1, 2, 4, 5])
@pytest.mark.parametrize("tile", [None, (16, 8), (128, 64), (128, 128)])
def test_fields_and_bins(torch_cuda, n_fields, tile):
    rng = np.random.default_rng(60 + n_fields)
    wl = synth.small_workload(60, 96, 48, n_fields=n_fields, dtype="f64", points="uniform")
    lon, colat = points(rng, 3001)
    vals, _ = values(torch_cuda, wl.coeffs, lon, colat, 96, 48, tile=tile)
    ref = oracle.evaluate(wl.coeffs, lon, colat)
    for f in range(n_fields):
        assert oracle.rel_linf(vals[f], ref[f].real) <= 1e-11


@pytest.mark.parametrize("scale", [1e-300, 1e-150, 1e-30, 1.0, 1e30, 1e200, 1e300])
def test_magnitudes_side_by_side(torch_cuda, scale):
    rng = np.random.default_rng(61)
    wl = synth.small_workload(61, 64, 32, n_fields=3, dtype="f64", points="uniform")
    c = wl.coeffs.copy()
    c[0] *= scale
    c[1] = 0.0
    lon, colat = points(rng, 2000)
    vals, _ = values(torch_cuda, c, lon, colat, 64, 32)
    ref = oracle.evaluate(wl.coeffs, lon, colat)
    assert oracle.rel_linf(vals[0] / scale, ref[0].real) <= 1e-11
    assert (vals[1] == 0.0).all()
    assert oracle.rel_linf(vals[2], ref[2].real) <= 1e-11


def test_steep_field(torch_cuda):
    """A field that is zero to rounding over most of the sphere: a bump whose tail
    falls far below the FP64 resolution of its peak."""
    c = synth.gaussian_bump_coeffs(128, 64, 1.0, 1.2, 8.0e5, 1.0)[None]
    rng = np.random.default_rng(62)
    lon, colat = points(rng, 3000)
    vals, _ = values(torch_cuda, c, lon, colat, 128, 64, real_fields=True)
    ref = oracle.evaluate(c, lon, colat)
    assert oracle.rel_linf(vals[0], ref[0].real) <= 1e-11


@pytest.mark.parametrize("bad", [math.nan, math.inf, -math.inf])
def test_non_finite_input(torch_cuda, bad):
    rng = np.random.default_rng(63)
    wl = synth.small_workload(63, 64, 32, n_fields=2, dtype="f64", points="uniform")
    c = wl.coeffs.copy()
    c[0, 5, 7] = bad
    lon, colat = points(rng, 1000)
    lon[::7] = bad
    colat[3::11] = bad
    vals, _ = values(torch_cuda, c, lon, colat, 64, 32)
    ok = np.isfinite(lon) & np.isfinite(colat)
    assert np.isnan(vals[0]).all()
    assert np.isnan(vals[1][~ok]).all()
    ref = oracle.evaluate(wl.coeffs[1:], lon[ok], colat[ok])
    assert oracle.rel_linf(vals[1][ok], ref[0].real) <= 1e-11
