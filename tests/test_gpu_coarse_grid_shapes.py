"""The smooth terms' coarse grid where a rank exceeds another mode's grid size: the split precisions run it
with modes 2 and 3 exchanged, so r3 takes the place of n2 and r2 that of n3.  Apply, energy and both gradients
against the oracle at the tolerances of the precisions' parity tests."""
import numpy as np
import pytest

import oracle as O
from _helpers import E_TOL, assert_close, to_gpu
from test_gpu_term_split import MIXED, system

pytestmark = pytest.mark.gpu

SHAPES = [
    ((24, 14, 120), (10, 11, 60)),      # r3 > n2
    ((20, 72, 16), (10, 40, 11)),       # r2 > n3
    ((12, 20, 44), (11, 10, 21)),       # r3 = n2 + 1
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


@pytest.mark.parametrize("prec", ["fp32", "tf32x3", "bf16x3"])
@pytest.mark.parametrize("n,r", SHAPES)
def test_ranks_above_another_modes_grid(n, r, prec):
    import paper_2401_04189_gb300 as P
    s = system(n, r, [t * 0.1 for t in MIXED])
    S = O.Setup.from_system(s)
    ctx = P.Context.from_system(s, precision=prec)
    occ = to_gpu(s.psi)
    ref = O.exchange_apply(s.psi, S)
    got, e = P.tx_exchange_apply_energy(ctx, occ)
    assert_close(got.cpu().numpy(), ref, prec, "coarse-shape")
    ref_e = O.exchange_energy(s.psi, S, W=ref)
    assert abs(float(e.item()) - ref_e) < E_TOL[prec] * abs(ref_e)
    _, grad = P.tx_exchange_energy_grad(ctx, occ)
    assert_close(grad.cpu().numpy(), O.exchange_energy_grad(s.psi, S)[1], prec, "coarse-shape-grad", scale=5)
    ctx.check_device_error()
