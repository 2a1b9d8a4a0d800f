"""set_points where its one-pass bin scan and its short angle reduction can go
wrong: many scan chunks with points in a few far-apart bins, bins at both ends
of the list, points on one side of the torus seam, members of very different
point counts, and angles on both sides of the magnitudes the short reduction
takes (2^-11 <= |v| < 2^9).

Reference: the FP64 oracle; bounds 1e-11 (FP64) and 2e-5 (FP32) as everywhere.
An angle v is resolved to its own rounding: the field's largest wavenumber (16
here) times the spacing of FP64 numbers at |v| bounds what the oracle's own
sine and cosine may add, 16 x 2^-34 = 1e-9 at |v| = 2^19 at most, so those
points are reduced to [0, 2 pi) in extended precision for the oracle."""
import math

import numpy as np
import pytest

import oracle
from paper_2605_01313_gb300 import build

pytestmark = pytest.mark.gpu

BOUND = {"f64": 1e-11, "f32": 2e-5}


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for the -m gpu tests")
    build.build()
    return torch


def sparse_coeffs(rng, F, n_lon, n_lat, k=16):
    """White noise in the modes |n|, |m| < k, zero elsewhere; and the small
    array of the same modes for the oracle."""
    c = np.zeros((F, 2 * n_lat, n_lon), dtype=np.complex128)
    small = rng.standard_normal((F, 2 * k, 2 * k)) + 1j * rng.standard_normal((F, 2 * k, 2 * k))
    small = small.astype(np.complex64).astype(np.complex128)
    small[:, 0, :] = small[:, :, 0] = 0.0
    c[:, n_lat - k:n_lat + k, n_lon // 2 - k:n_lon // 2 + k] = small
    return c, small


def values(torch, dtype, n_lon, n_lat, c, pts):
    from paper_2605_01313_gb300 import Plan
    cd = torch.complex128 if dtype == "f64" else torch.complex64
    M = len(pts)
    with Plan(n_lon, n_lat, 1e-12 if dtype == "f64" else 1e-6, dtype, c.shape[0],
              n_members=M) as plan:
        lon = torch.from_numpy(np.concatenate([p[0] for p in pts])).cuda()
        colat = torch.from_numpy(np.concatenate([p[1] for p in pts])).cuda()
        plan.set_points(lon, colat, [p[0].size for p in pts])
        co = torch.from_numpy(c).to(cd).cuda()
        out = plan.execute(co if M == 1 else co.expand(M, *co.shape).contiguous())
        plan.check()
        if M == 1:
            return [out.cpu().numpy()]
        return [v.cpu().numpy() for v in plan.split_values(out)]


def check(vals, small, lon, colat, bound):
    ref = oracle.evaluate(small, lon, colat)
    for f in range(small.shape[0]):
        assert oracle.rel_linf(vals[f], ref[f].real) <= bound


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("where", ["corners", "seam", "one", "rows", "everywhere"])
def test_scan_with_points_in_few_bins(torch_cuda, where, dtype):
    rng = np.random.default_rng(41)
    n_lon, n_lat = 1024, 512
    if where == "corners":               # first and last bins of the list
        lon = np.concatenate([rng.uniform(0, 0.01, 70), rng.uniform(6.27, 6.283, 90)])
        colat = np.concatenate([rng.uniform(0, 0.01, 70), rng.uniform(-0.01, 0, 90)])
    elif where == "seam":                # negative colatitudes: the other half of the torus
        lon, colat = rng.uniform(-0.05, 0.05, 1500), rng.uniform(-0.05, 0.05, 1500)
    elif where == "one":
        lon, colat = np.array([3.0]), np.array([2.0])
    elif where == "rows":                # few bin rows, far apart
        lon = rng.uniform(0, 2 * math.pi, 900)
        colat = np.repeat([0.1, 1.7, 1.8], 300) + rng.uniform(0, 1e-3, 900)
    else:                                # every bin of both halves
        lon, colat = rng.uniform(0, 2 * math.pi, 200001), rng.uniform(-math.pi, math.pi, 200001)
    c, small = sparse_coeffs(rng, 2, n_lon, n_lat)
    vals = values(torch_cuda, dtype, n_lon, n_lat, c, [(lon, colat)])
    pick = np.arange(lon.size) if lon.size < 2000 else np.sort(rng.choice(lon.size, 2000, False))
    check(vals[0][:, pick], small, lon[pick], colat[pick], BOUND[dtype])


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_scan_of_uneven_members(torch_cuda, dtype):
    rng = np.random.default_rng(42)
    c, small = sparse_coeffs(rng, 1, 512, 256)
    pts = [(rng.uniform(0, 2 * math.pi, n), rng.uniform(lo, hi, n))
           for n, lo, hi in ((1, 1.0, 1.1), (40000, 0.0, math.pi), (33, 3.0, 3.1),
                             (257, -0.2, 0.2))]
    vals = values(torch_cuda, dtype, 512, 256, c, pts)
    for v, (lon, colat) in zip(vals, pts):
        check(v[:, :1000], small, lon[:1000], colat[:1000], BOUND[dtype])


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_angles_on_both_sides_of_the_short_reduction(torch_cuda, dtype):
    rng = np.random.default_rng(43)
    mag = np.concatenate([2.0 ** -11 * (1 + rng.uniform(-1e-3, 1e-3, 40)),
                          512.0 * (1 + rng.uniform(-1e-3, 1e-3, 40)),
                          [2.0 ** -11, 512.0, np.nextafter(512.0, 0), np.nextafter(2.0 ** -11, 0),
                           0.0, 1e-300, 2.0 ** -60, 2.0 ** 19, 1000.0],
                          np.exp(rng.uniform(math.log(1e-9), math.log(2.0 ** 19), 200)),
                          np.arange(0, 64) * (2 * math.pi / 64)])
    lon = mag * rng.choice([-1.0, 1.0], mag.size)
    colat = rng.permutation(mag) * rng.choice([-1.0, 1.0], mag.size)
    c, small = sparse_coeffs(rng, 1, 128, 64)
    vals = values(torch_cuda, dtype, 128, 64, c, [(lon, colat)])
    # 2 pi in two parts: v - q 2 pi to a few 1e-17 for |q| < 2^17
    two_pi_hi, two_pi_lo = 2 * math.pi, 2.4492935982947064e-16

    def reduced(v):
        q = np.floor(v.astype(np.longdouble) / np.longdouble(two_pi_hi))
        r = v.astype(np.longdouble) - q * np.longdouble(two_pi_hi) - q * np.longdouble(two_pi_lo)
        return r.astype(np.float64)

    check(vals[0], small, reduced(lon), reduced(colat), BOUND[dtype])
