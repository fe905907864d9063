"""Mesh to grid in chunks of orbitals: a block gives, bit for bit, what its orbitals give a few at a time, at the edges
of the chunks (whole blocks, 8, 64 and 128 orbitals at a time, remainders), for every mesh order."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


@pytest.mark.parametrize("order,n,counts", [
    (1, (21, 22, 23), (1, 3, 8, 257, 300)),          # whole blocks, up to 256 orbitals
    (1, (101, 97, 90), (28, 29, 33, 50)),            # more than 100 MB: 8 at a time
    (2, (31, 40, 25), (1, 63, 65, 129)),
    (3, (31, 40, 25), (5, 127, 129, 260)),
])
def test_chunks_agree_with_few_orbitals(order, n, counts):
    import paper_2401_04189_gb300 as P
    xs = [np.linspace(-4.0, 4.0, k) for k in n]
    ctx = P.Context(xs, [np.ones(k) for k in n], [np.eye(k)[:, :1] for k in n], [1.0], [1.0], precision="fp32")
    X, conn = W.fe_mesh(4.0, 3, np.array([[0.5, -1.0, 2.0], [-2.0, 1.5, -0.5]]), 1.2, order)
    tr = P.Transfer(ctx, X, conn, order, 1)
    gen = torch.Generator(device="cuda").manual_seed(order)
    psi = torch.randn((X.shape[0], max(counts)), generator=gen, device="cuda")
    few = torch.cat([tr.u_to_s(psi[:, k:k + 4].contiguous()) for k in range(0, max(counts), 4)])
    for c in counts:
        got = tr.u_to_s(psi[:, :c].contiguous(), out=torch.full((c, *n), float("nan"), device="cuda"))
        assert torch.equal(got, few[:c])
