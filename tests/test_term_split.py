"""The rule that sends a Gaussian term to the coarse grid (CPU): for every exponent the bound admits,
Chebyshev interpolation of exp(-theta (x - c)^2) with that many nodes is accurate to the tolerance,
wherever the centre lies."""
import math

import numpy as np
import pytest

TOL = 1e-9


def bound(theta, h, N):
    a = theta * h * h
    eta = 0.5 * math.asinh(N / a)
    return 4.0 * math.exp(a * math.sinh(eta) ** 2 - N * eta) / (math.exp(eta) - 1.0)


@pytest.mark.parametrize("r", [6, 13, 16, 40, 64])
@pytest.mark.parametrize("h", [0.7, 12.0])
def test_admitted_exponents_interpolate_to_the_tolerance(r, h):
    lo, hi = 1e-12 / h ** 2, 1e4 / h ** 2            # the largest exponent that the bound admits
    assert bound(lo, h, r - 1) <= TOL
    for _ in range(60):
        mid = math.sqrt(lo * hi)
        lo, hi = (mid, hi) if bound(mid, h, r - 1) <= TOL else (lo, mid)
    k = np.arange(r)
    xi = -h * np.cos(np.pi * (k + 0.5) / r)
    w = np.where(k % 2, -1.0, 1.0) * np.sin(np.pi * (k + 0.5) / r)
    x = np.linspace(-h, h, 301)
    d = x[:, None] - xi[None, :]
    d[d == 0] = 1e-300
    L = w / d
    L /= L.sum(1, keepdims=True)
    for c in np.concatenate([np.linspace(-h, h, 23), [-1.4 * h, 2.0 * h]]):
        for theta in (lo, lo / 3, lo / 100):
            err = np.abs(L @ np.exp(-theta * (xi - c) ** 2) - np.exp(-theta * (x - c) ** 2)).max()
            assert err <= TOL
    assert bound(2.0 * lo, h, r - 1) > TOL
