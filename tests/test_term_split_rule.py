"""The library's own rule for the terms on the coarse grid (tx_describe_term_split, host only): the largest exponent
that it admits, found by bisection, interpolates exp(-theta (x - c)^2) to 1e-9 wherever the centre lies, twice that
exponent is not admitted; every mode counts; and the split runs where it saves work and only there."""
import math

import numpy as np
import pytest

import paper_2401_04189_gb300 as P
from test_gpu_term_split import CASES, system

EXPECTED = {"mixed": 4, "graded": 4, "smooth": 5, "sharp": 0, "two": 2}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


def admits(theta, h, r, n=256):
    return P.tx_describe_term_split((n,) * 3, (r,) * 3, (2 * h,) * 3, [theta])[0][0]


def largest(h, r):
    lo, hi = 1e-12 / h ** 2, 1e5 / h ** 2
    assert admits(lo, h, r) and not admits(hi, h, r)
    for _ in range(60):
        mid = math.sqrt(lo * hi)
        lo, hi = (mid, hi) if admits(mid, h, r) else (lo, mid)
    return lo


@pytest.mark.parametrize("r", [6, 13, 16, 40, 64])
@pytest.mark.parametrize("h", [0.7, 12.0])
def test_admitted_exponents_interpolate_to_the_tolerance(r, h):
    top = largest(h, r)
    assert not admits(2.0 * top, h, r)
    k = np.arange(r)
    xi = -h * np.cos(np.pi * (k + 0.5) / r)
    w = np.where(k % 2, -1.0, 1.0) * np.sin(np.pi * (k + 0.5) / r)
    x = np.linspace(-h, h, 301)
    d = x[:, None] - xi[None, :]
    d[d == 0] = 1e-300
    L = w / d
    L /= L.sum(1, keepdims=True)
    for c in np.concatenate([np.linspace(-h, h, 23), [-1.4 * h, 2.0 * h]]):
        for theta in (top, top / 3, top / 100):
            assert np.abs(L @ np.exp(-theta * (xi - c) ** 2) - np.exp(-theta * (x - c) ** 2)).max() <= 1e-9


def test_the_mode_with_the_fewest_nodes_decides():
    top = largest(5.0, 20)
    for d in range(3):
        r, ext = [40, 40, 40], [10.0, 10.0, 10.0]
        r[d] = 20
        assert P.tx_describe_term_split((256,) * 3, r, ext, [top, 2 * top])[0] == [True, False]
        ext[d] = 20.0                          # twice the length: a quarter of the exponent
        assert P.tx_describe_term_split((256,) * 3, r, ext, [top, 0.25 * top])[0] == [False, True]
    assert P.tx_describe_term_split((8, 8, 8), (1, 4, 4), (1.0,) * 3, [1e-9])[0] == [False]      # one node


@pytest.mark.parametrize("case", sorted(CASES))
def test_terms_of_the_parity_cases(case):
    n, r, theta, uniform = CASES[case]
    s = system(n, r, theta, uniform=uniform, n_orb=1)
    extent = [float(x.max() - x.min()) for x in s.x]
    smooth, coarse = P.tx_describe_term_split(n, r, extent, theta)
    assert (sum(smooth), coarse) == (EXPECTED[case], EXPECTED[case])


def test_no_coarse_grid_where_it_saves_nothing():
    smooth, coarse = P.tx_describe_term_split((16, 16, 16), (16, 16, 16), (1.0,) * 3, [1e-6] * 8)
    assert all(smooth) and coarse == 0         # full rank: the coarse grid is as large
    smooth, coarse = P.tx_describe_term_split((64, 64, 64), (16, 16, 16), (1.0,) * 3, [1e-6])
    assert all(smooth) and coarse == 0         # one term: the interpolation costs as much
    assert P.tx_describe_term_split((64, 64, 64), (16, 16, 16), (1.0,) * 3, [1e-6] * 2)[1] == 2


@pytest.mark.parametrize("args,status", [
    (((64,) * 3, (16,) * 3, (1.0,) * 3, [0.0]), -1), (((64,) * 3, (16,) * 3, (1.0,) * 3, [-1.0]), -1),
    (((64,) * 3, (16,) * 3, (float("nan"), 1.0, 1.0), [1.0]), -1), (((64,) * 3, (16,) * 3, (1.0,) * 3, []), -1),
    (((1, 64, 64), (1, 16, 16), (1.0,) * 3, [1.0]), -2), (((64,) * 3, (65, 16, 16), (1.0,) * 3, [1.0]), -2)])
def test_bad_arguments(args, status):
    with pytest.raises(P.TuckerExchangeError) as e:
        P.tx_describe_term_split(*args)
    assert e.value.status == status
