"""The split precisions' operand image serves every tile plan that a caller can force: whole slabs of one and more
planes, the operand in shared memory and in tensor memory, and y/z items (where no whole-slab plan is accepted).
Against the oracle, at the precisions' tolerances."""
import pytest

import oracle as O
from _helpers import assert_close, to_gpu
from test_gpu_term_split import system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
@pytest.mark.parametrize("n,r", [((12, 40, 32), (6, 13, 11)), ((10, 90, 40), (5, 20, 17)), ((6, 130, 48), (4, 24, 18)),
                                 ((4, 200, 200), (3, 33, 41))])
def test_every_forced_plan_agrees(n, r, prec):
    import paper_2401_04189_gb300 as P
    s = system(n, r, [3.0, 0.05, 12.0], n_orb=2)
    ref = O.exchange_apply(s.psi, O.Setup.from_system(s))
    ctx = P.Context.from_system(s, precision=prec)
    occ = to_gpu(s.psi)
    for bx in (0, 1, 2, 3, 6):
        for ns in ((0,) if bx == 0 else (1, 2, 4)):
            try:
                P.tx_set_tile_plan(ctx, bx, ns)
            except P.TuckerExchangeError:
                continue                      # does not fit this shape
            got = P.tx_exchange_apply(ctx, occ).cpu().numpy()
            ctx.check_device_error()
            assert_close(got, ref, prec, f"split-plan-{bx}-{ns}")
