"""Smooth Gaussian terms on the coarse Chebyshev grid, against the oracle (which sums every term on
the fine grid): mixed, only smooth and only sharp exponents, in any order; non-uniform grids; ranks
that differ per mode; finite-element quadrature; apply, energy, both gradients and the
allocation-free apply.  Tolerances are those of the precisions' parity tests."""
import math

import numpy as np
import pytest

import oracle as O
import workloads as W
from _helpers import E_TOL, assert_close, to_gpu

pytestmark = pytest.mark.gpu

MIXED = [30.0, 0.004, 2.5, 0.02, 1e-5, 0.3, 8.0, 0.0007, 0.05, 1e-3]      # not sorted
SMOOTH = [0.01, 1e-4, 0.002, 3e-6, 0.0005, 0.004]
SHARP = [3.0, 12.0, 40.0]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


def system(n, r, theta, seed=11, n_orb=3, uniform=True):
    rng = np.random.default_rng(seed)
    half = [0.15 * (k - 1) for k in n]
    xs, ws = [], []
    for k, L in zip(n, half):
        x, w = W.uniform_grid(k, L)
        if not uniform:                      # graded and shifted, trapezoid weights
            x = L * np.sinh(1.3 * x / L) / math.sinh(1.3) + 0.4
            d = np.diff(x)
            w = np.concatenate([[d[0]], d[:-1] + d[1:], [d[-1]]]) / 2
        xs.append(x)
        ws.append(w)
    cen = rng.uniform(-1.0, 1.0, size=(n_orb, 3, 3))
    psi = W.gaussian_sum_orbitals(xs, cen, rng.uniform(0.3, 1.5, (n_orb, 3)), rng.standard_normal((n_orb, 3)))
    psi = W.lowdin_orthonormalise(psi, ws).astype(np.float32)
    U = W.density_hosvd_basis(psi, r)
    mu = rng.uniform(0.2, 1.0, len(theta)) * np.sqrt(np.asarray(theta))
    return W.System("split", xs, ws, U, np.asarray(theta, dtype=np.float64), mu, psi, 0.0)


CASES = {
    "mixed": ((30, 36, 40), (12, 13, 16), MIXED, True),
    "graded": ((28, 33, 44), (14, 12, 15), MIXED, False),
    "smooth": ((31, 29, 36), (11, 14, 13), SMOOTH, True),
    "sharp": ((24, 26, 28), (10, 9, 12), SHARP, True),
    "two": ((32, 32, 32), (12, 12, 12), [0.003, 9.0, 0.0002], True),
}


def check_all(s, S, ctx, prec):
    import paper_2401_04189_gb300 as P
    occ = to_gpu(s.psi)
    ref = O.exchange_apply(s.psi, S)
    got, e = P.tx_exchange_apply_energy(ctx, occ)
    assert_close(got.cpu().numpy(), ref, prec, "split")
    ref_e = O.exchange_energy(s.psi, S, W=ref)
    assert abs(float(e.item()) - ref_e) < E_TOL[prec] * abs(ref_e)
    assert_close(P.tx_exchange_apply(ctx, occ, occ[1:2]).cpu().numpy(), ref[1:2], prec, "split-slice")
    _, grad = P.tx_exchange_energy_grad(ctx, occ)
    assert_close(grad.cpu().numpy(), O.exchange_energy_grad(s.psi, S)[1], prec, "split-grad", scale=5)
    rng = np.random.default_rng(2)
    tgt, cot = rng.standard_normal((2, 2, *s.psi.shape[1:])).astype(np.float32)
    ro, rt = O.exchange_apply_vjp(s.psi, tgt, cot, S)
    go, gt = P.tx_exchange_apply_vjp(ctx, occ, to_gpu(tgt), to_gpu(cot))
    assert_close(go.cpu().numpy(), ro, prec, "split-vjp-occ", scale=5)
    assert_close(gt.cpu().numpy(), rt, prec, "split-vjp-tgt", scale=5)
    ctx.check_device_error()


@pytest.mark.parametrize("prec", ["fp32", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("case", sorted(CASES))
def test_split_matches_oracle(case, prec):
    import paper_2401_04189_gb300 as P
    n, r, theta, uniform = CASES[case]
    s = system(n, r, theta, uniform=uniform)
    check_all(s, O.Setup.from_system(s), P.Context.from_system(s, precision=prec), prec)


@pytest.mark.parametrize("prec", ["fp32", "tf32x3"])
def test_split_follows_the_quadrature(prec):
    import paper_2401_04189_gb300 as P
    s = system((31, 37, 40), (13, 12, 14), MIXED)
    ctx = P.Context.from_system(s, precision=prec)
    ctx.set_quadrature(3, 4)
    check_all(s, O.Setup.from_system(s, quadrature=("fe", 3, 4)), ctx, prec)
    ctx.set_quadrature(0)
    check_all(s, O.Setup.from_system(s), ctx, prec)


def test_static_apply_uses_the_same_terms():
    import torch
    import paper_2401_04189_gb300 as P
    from paper_2401_04189_gb300 import _lib
    s = system((30, 36, 40), (12, 13, 16), MIXED)
    ctx = P.Context.from_system(s, precision="fp32")
    occ, out = to_gpu(s.psi), torch.empty_like(to_gpu(s.psi))
    assert P.lib().tx_exchange_apply_static(ctx.handle, _lib._ptr(occ), occ.shape[0], _lib._ptr(out), _lib._stream(None)) == 0
    assert_close(out.cpu().numpy(), O.exchange_apply(s.psi, O.Setup.from_system(s)), "fp32", "split-static")
