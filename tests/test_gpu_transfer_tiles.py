"""Mesh-to-grid transfer at the edges of its tiles, against the oracle: cells of one to several blocks of
nodes, blocks that fill one to four nodes per thread with a remainder, one orbital, a remainder of four and
more orbitals than one staged chunk.  Random nodal values; the sum of at most 64 products in float32 stays
within 64 x 2^-24 times the sum of the magnitudes, 4e-6 of the largest value times the Lebesgue constant
(below 2 per mode for these nodes); random signs keep it below 1e-6 as in the parity test."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


@pytest.mark.parametrize("order_u", [1, 2, 3])
@pytest.mark.parametrize("n,n_orb", [((3, 2, 5), 1), ((11, 10, 9), 6), ((13, 14, 15), 131), ((34, 31, 37), 5)])
def test_blocks_of_a_cell(n, n_orb, order_u):
    import torch
    import paper_2401_04189_gb300 as P
    xs, ws = zip(*[W.uniform_grid(k, 2.0) for k in n])
    ctx = P.Context(list(xs), list(ws), [np.eye(k)[:, :1] for k in n], [1.0], [1.0], precision="fp32")
    X, conn = W.fe_mesh(2.0, 2, np.zeros((1, 3)), 0.0, order_u, levels=0)
    psi_u = np.random.default_rng(1).standard_normal((len(X), n_orb)).astype(np.float32)
    tr = P.Transfer(ctx, X, conn, order_u, 1)
    got = tr.u_to_s(torch.from_numpy(psi_u).cuda()).cpu().numpy()
    ref = O.transfer_u_to_s(psi_u.astype(np.float64), X, conn, order_u, list(xs))
    assert np.max(np.abs(got - ref)) < 1e-6 * np.max(np.abs(ref))
    tr.destroy()
