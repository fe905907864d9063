"""Split precisions (TF32x3, BF16x3) at the edges of the expansion kernel's tiles, against the oracle:
the converted operand in shared memory (n2 <= 64) and in tensor memory (above), one and two y tiles
with a remainder, several planes per CTA, (y, z) parts, and ranks that fill neither a group of 8 nor
an MMA's K.  The exponents are too sharp for the coarse grid, so every term runs on the fine one.
Tolerances are those of the precisions' parity tests.  The two-sided projection of one and two pairs,
whose terms are split over CTAs, is held to the float32 ones."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from _helpers import assert_close, to_gpu

pytestmark = pytest.mark.gpu

SHAPES = [
    ((9, 12, 20), (4, 5, 9)),
    ((5, 64, 24), (4, 13, 11)),
    ((5, 65, 24), (4, 13, 11)),
    ((3, 128, 32), (3, 17, 9)),
    ((3, 129, 32), (2, 20, 24)),
    ((2, 30, 200), (2, 12, 41)),
    ((4, 200, 40), (3, 33, 18)),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


def _system(n, r, theta, n_orb, seed=5):
    rng = np.random.default_rng(seed)
    xs, ws = zip(*[W.uniform_grid(k, 2.0) for k in n])
    psi = rng.standard_normal((n_orb, *n)).astype(np.float32)
    U = [np.linalg.qr(rng.standard_normal((k, q)))[0] for k, q in zip(n, r)]
    theta = np.asarray(theta, dtype=np.float64)
    return W.System("tiles", list(xs), list(ws), U, theta, 0.3 + 0.1 * np.sqrt(theta), psi, 0.0)


@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
@pytest.mark.parametrize("n,r", SHAPES)
def test_split_apply(n, r, prec):
    import paper_2401_04189_gb300 as P
    s = _system(n, r, [40.0, 90.0, 25.0, 300.0, 60.0], 3)
    ctx = P.Context.from_system(s, precision=prec)
    got = P.tx_exchange_apply(ctx, to_gpu(s.psi))
    assert_close(got.cpu().numpy(), O.exchange_apply(s.psi, O.Setup.from_system(s)), prec, "tiles")


@pytest.mark.parametrize("n_orb,T", [(1, 3), (1, 8), (1, 9), (2, 23), (2, 40)])
@pytest.mark.parametrize("r", [(1, 2, 3), (7, 9, 8), (13, 18, 23)])
def test_two_sided_terms_over_ctas(r, n_orb, T):
    import paper_2401_04189_gb300 as P
    s = _system((14, 19, 24), r, np.geomspace(0.01, 50.0, T), n_orb)
    ctx = P.Context.from_system(s, precision="fp32")
    got = P.tx_exchange_apply_galerkin(ctx, to_gpu(s.psi))
    assert_close(got.cpu().numpy(), O.exchange_apply_galerkin(s.psi, O.Setup.from_system(s)), "fp32", "tiles-galerkin", scale=5)
