"""Expansion plans within a few KB of the shared-memory limit against the oracle, at the tolerances of the
precisions' parity tests: each kernel form of the converter (operand in shared memory and in tensor memory,
single-pass and split, whole slabs and y/z items)."""
import pytest

import oracle as O
from _helpers import assert_close, to_gpu
from test_gpu_term_split import system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


@pytest.mark.parametrize("prec,n,r", [
    ("tf32", (40, 192, 84), (20, 89, 71)),
    ("bf16", (51, 215, 128), (45, 190, 108)),
    ("tf32x3", (20, 60, 232), (16, 40, 128)),
    ("bf16x3", (60, 223, 136), (33, 185, 95)),
    ("tf32x3", (41, 162, 216), (41, 131, 72)),
])
def test_plans_near_the_limit(prec, n, r):
    import paper_2401_04189_gb300 as P
    s = system(n, r, [0.6, 0.02, 3.0, 9.0], n_orb=2)
    ctx = P.Context.from_system(s, precision=prec)
    got = P.tx_exchange_apply(ctx, to_gpu(s.psi)).cpu().numpy()
    ctx.check_device_error()
    assert_close(got, O.exchange_apply(s.psi, O.Setup.from_system(s)), prec, "plan-limit")
