"""The one-launch set_points of small members against the general path of larger
ones at the edges of its range: 4096 points a member (the largest it takes) and
4097, one point, members of unlike counts, 8192 rows of bins and more, in both
precisions and with points everywhere, in one bin and at the torus seam.

Reference: the FP64 oracle; bounds 1e-11 (FP64) and 2e-5 (FP32) as everywhere."""
import math

import numpy as np
import pytest

from test_points_scan_gpu import BOUND, check, sparse_coeffs, torch_cuda, values  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("n_points", [1, 31, 1023, 1025, 4096, 4097])
@pytest.mark.parametrize("n_lon,n_lat", [(64, 32), (128, 64), (256, 128), (512, 128), (64, 512)])
def test_edges_of_the_range(torch_cuda, n_lon, n_lat, n_points, dtype):  # noqa: F811
    rng = np.random.default_rng(n_points + n_lon)
    c, small = sparse_coeffs(rng, 2, n_lon, n_lat)
    lon, colat = rng.uniform(-1, 7, n_points), rng.uniform(-math.pi, math.pi, n_points)
    vals = values(torch_cuda, dtype, n_lon, n_lat, c, [(lon, colat)])
    check(vals[0], small, lon, colat, BOUND[dtype])


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("counts", [(1, 4096, 33, 700), (4097, 5, 64)])
def test_members(torch_cuda, counts, dtype):  # noqa: F811
    rng = np.random.default_rng(sum(counts))
    c, small = sparse_coeffs(rng, 1, 64, 32)
    pts = [(rng.uniform(0, 2 * math.pi, n), rng.uniform(0, math.pi, n)) for n in counts]
    for v, (lon, colat) in zip(values(torch_cuda, dtype, 64, 32, c, pts), pts):
        check(v, small, lon, colat, BOUND[dtype])


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("where", ["one_bin", "seam", "two_rows"])
def test_clustered_points(torch_cuda, where, dtype):  # noqa: F811
    rng = np.random.default_rng(9)
    n = 3000
    lon, colat = {"one_bin": (rng.uniform(1.0, 1.01, n), rng.uniform(1.0, 1.01, n)),
                  "seam": (rng.uniform(-0.02, 0.02, n), rng.uniform(-0.02, 0.02, n)),
                  "two_rows": (rng.uniform(0, 6.28, n), rng.choice([0.1, 3.0], n))}[where]
    c, small = sparse_coeffs(rng, 2, 64, 32)
    vals = values(torch_cuda, dtype, 64, 32, c, [(lon, colat)])
    check(vals[0], small, lon, colat, BOUND[dtype])
