"""M_ij = <psi_i, W_j>_w across chunks of 64 grid points is a float64 sum of the chunks' float32 sums: chunk sums
-1, -2^27, -1, 2^27 add up to -2 exactly, whatever a float32 total makes of them.  One and several output tiles,
slices of few chunks and of more than one float64 addition takes (64 chunks).  Every product and every chunk sum is
exact, so M has to be equal to the integers."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


@pytest.mark.parametrize("n,N", [((16, 16, 16), 1), ((16, 16, 16), 17), ((24, 20, 16), 33), ((20, 20, 21), 64),
                                 ((56, 56, 56), 130)])
def test_chunk_sums_that_cancel(n, N):
    import paper_2401_04189_gb300 as P
    xs = [np.arange(k, dtype=np.float64) for k in n]
    ctx = P.Context(xs, [np.ones(k) for k in n], [np.eye(k)[:, :1] for k in n], [1.0], [1.0], precision="fp32")
    N3 = n[0] * n[1] * n[2]
    classes = (N + 63) // 64                  # orbital i lives at offset i % 64 of every classes-th four chunks
    psi = torch.zeros((N, N3), device="cuda")
    W = torch.zeros((N, N3), device="cuda")
    quads = N3 // 256
    chunk = torch.tensor([-1.0, -2.0 ** 27, -1.0, 2.0 ** 27], device="cuda")
    expect = np.zeros(N)
    for i in range(N):
        q = torch.arange(i // 64, quads, classes, device="cuda")
        at = (256 * q[:, None] + 64 * torch.arange(4, device="cuda")[None, :] + i % 64).reshape(-1)
        psi[i, at] = 1.0
        W[i, at] = chunk.repeat(len(q))
        expect[i] = -2.0 * len(q)
    _, M = P.tx_ace_projectors(ctx, psi.reshape(N, *n), W.reshape(N, *n))
    assert np.array_equal(M.cpu().numpy(), np.diag(expect))
