"""V_ACE psi = - sum_k xi_k <xi_k, psi>_w at the edges of the Gram kernel's tiles (16, 32 and 64 orbitals per
side, one and more tiles, slices that end inside a chunk, grids without 16-byte rows) against numpy in
float64.  Bound: the Gram matrix and the mix each round like one float32 product (4 unit roundoffs of the
sum of the magnitudes).  An infinite orbital value gives infinite or NaN output, not a finite one."""
import numpy as np
import pytest

import workloads as W
from _helpers import to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


def _context(n):
    import paper_2401_04189_gb300 as P
    xs, ws = zip(*[W.uniform_grid(k, 2.0) for k in n])
    return P.Context(list(xs), list(ws), [np.eye(k)[:, :1] for k in n], [1.0], [1.0], precision="fp32"), ws


@pytest.mark.parametrize("n", [(5, 7, 9), (16, 24, 20)])
@pytest.mark.parametrize("nxi,npsi", [(1, 1), (16, 33), (17, 16), (64, 65), (70, 5), (32, 64)])
def test_ace_apply_tiles(n, nxi, npsi):
    import paper_2401_04189_gb300 as P
    ctx, ws = _context(n)
    rng = np.random.default_rng(nxi * 100 + npsi)
    xi = rng.standard_normal((nxi, *n)).astype(np.float32)
    psi = rng.standard_normal((npsi, *n)).astype(np.float32)
    got = P.tx_ace_apply(ctx, to_gpu(xi), to_gpu(psi)).cpu().numpy().reshape(npsi, -1)
    w = np.einsum("i,j,k->ijk", *ws).reshape(-1)
    x, p = xi.reshape(nxi, -1).astype(np.float64), psi.reshape(npsi, -1).astype(np.float64)
    ref = -((p * w) @ x.T) @ x
    mag = ((np.abs(p) * w) @ np.abs(x).T) @ np.abs(x)
    assert np.all(np.abs(got - ref) <= 4 * 2.0 ** -24 * mag)


def test_infinite_value_does_not_turn_finite():
    import paper_2401_04189_gb300 as P
    n = (16, 24, 20)
    ctx, _ = _context(n)
    rng = np.random.default_rng(0)
    xi = np.abs(rng.standard_normal((3, *n))).astype(np.float32)
    psi = np.abs(rng.standard_normal((2, *n))).astype(np.float32)
    psi[1, 0, 0, 0] = np.inf
    got = P.tx_ace_apply(ctx, to_gpu(xi), to_gpu(psi)).cpu().numpy()
    assert np.isfinite(got[0]).all()
    assert np.isneginf(got[1]).all()
