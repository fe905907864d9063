"""BF16x3 where the smooth terms carry nearly all of W: they are summed and expanded in float32, so the error is that of
the float32 precision on the same inputs (twice it: another order of the same sums) plus the precision's own tolerance
on the sharp term's share of W.  Apply with the targets inside and beside the block, energy and gradient."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from _helpers import E_TOL, W_TOL, rel, to_gpu
from test_gpu_term_split import system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


@pytest.mark.parametrize("n,r", [((30, 36, 40), (12, 13, 16)), ((20, 70, 44), (10, 20, 15)), ((12, 140, 36), (9, 30, 14))])
def test_smooth_terms_keep_float32(n, r):
    import paper_2401_04189_gb300 as P
    s = system(n, r, [0.005, 0.002, 9.0, 0.0002, 0.001])
    s.mu[2] *= 1e-4
    extent = [float(x.max() - x.min()) for x in s.x]
    assert P.tx_describe_term_split(n, r, extent, s.theta) == ([True, True, False, True, True], 4)
    S = O.Setup.from_system(s)
    ref, ref_e = O.exchange_apply(s.psi, S), O.exchange_energy(s.psi, S)
    ref_grad = O.exchange_energy_grad(s.psi, S)[1]
    sharp = O.Setup.from_system(dataclasses.replace(s, theta=s.theta[2:3], mu=s.mu[2:3]))
    share = rel(ref + O.exchange_apply(s.psi, sharp), ref)       # |W_sharp| / |W|
    occ = to_gpu(s.psi)
    errs = {}
    for prec in ("fp32", "bf16x3"):
        ctx = P.Context.from_system(s, precision=prec)
        got, e = P.tx_exchange_apply_energy(ctx, occ)
        _, grad = P.tx_exchange_energy_grad(ctx, occ)
        errs[prec] = [rel(got.cpu().numpy(), ref), rel(P.tx_exchange_apply(ctx, occ, occ[1:2]).cpu().numpy(), ref[1:2]),
                      rel(P.tx_exchange_apply(ctx, occ, occ[:2].clone()).cpu().numpy(), ref[:2]),
                      rel(grad.cpu().numpy(), ref_grad)]
        ctx.check_device_error()
        for v in (float(e.item()), float(P.tx_exchange_energy(ctx, occ).item())):
            assert abs(v - ref_e) < E_TOL[prec] * abs(ref_e)
    for a, b in zip(errs["bf16x3"], errs["fp32"]):
        assert a < 2 * b + 2 * share * W_TOL["bf16x3"], (errs, share)
