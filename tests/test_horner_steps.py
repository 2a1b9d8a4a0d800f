"""The leading Horner steps that the FP64 interpolation takes in plain FP32 (no GPU):
for every kernel width and both oversampling factors, their rounding and the low
parts they leave out change a weight by less than 5e-16 of the largest one (which is
1), an eighth of the rounding of double-single arithmetic (2^-48 = 3.6e-15)."""
import math

import numpy as np
import pytest

from paper_2605_01313_gb300 import build, nufft


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


def plain_step_error(w, beta, steps):
    """Largest change of any tap's weight over |s| <= 1/2: `steps` FP32 fused
    multiply-adds in u = s^2 against FP64, in the even and the odd chain, each
    carried through the steps that remain (exactly: times u a step)."""
    P = nufft.dfsnufft_es_horner(w, beta)
    f32, f64 = np.float32, np.float64
    s = np.linspace(0.0, 0.5, 4001)
    u = s * s
    u_hi = u.astype(f32).astype(f64)
    worst = 0.0
    for a in range((w + 1) // 2):
        total = np.zeros_like(s)
        for k0, k1, scale in ((w - (w & 1), 0, 1.0), (w - 1 + (w & 1), 1, s)):
            approx, exact, k = np.full(u.shape, f64(f32(P[a, k0]))), np.full(u.shape, P[a, k0]), k0
            for _ in range(steps):
                if k - 2 < k1:
                    break
                k -= 2
                approx = (approx * u_hi + f64(f32(P[a, k]))).astype(f32).astype(f64)
                exact = exact * u + P[a, k]
            if steps:
                total += np.abs(approx - exact) * u ** ((k - k1) // 2) * scale
        worst = max(worst, float(total.max()))
    return worst


@pytest.mark.parametrize("sigma", [2, 4])
@pytest.mark.parametrize("w", range(2, 17))
def test_plain_steps_stay_below_double_single(w, sigma):
    beta = 2.30 * w if sigma == 2 else 0.97 * math.pi * (1 - 1 / 8) * w
    steps = nufft.dfsnufft_probe_plain_horner_steps(w)
    assert plain_step_error(w, beta, steps) <= 5e-16
