"""Per-pair bases where the Gram matrices have clustered or repeated eigenvalues: densities that are sums of products
of orthonormal vectors, sum_k s_k u_k x v_k x w_k, so every unfolding's Gram matrix has the eigenvalues s_k^2.  The
ranks cut at a gap of nearly the largest eigenvalue, where the projectors are well defined, and the one exponent is
so sharp that C is diagonal: phi is the projected density.  Bound: a mode's Gram matrix is a float32 sum of K
products (K = the other two sizes), so its projector is off by at most K 2^-24 over a gap of 1; three modes."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from _helpers import rel, to_gpu

pytestmark = pytest.mark.gpu

SPECTRA = {
    "repeated": np.concatenate([np.ones(10), 1e-3 * np.ones(6)]),
    "tight": np.concatenate([1 + 1e-6 * np.arange(10), 1e-4 * (1 + 1e-6 * np.arange(6))]),
    "clusters": np.concatenate([1 + 1e-3 * np.arange(6), 1.5 + 1e-5 * np.arange(4), 1e-3 * (1 + 1e-2 * np.arange(6))]),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


@pytest.mark.parametrize("n", [(49, 24, 17), (16, 64, 33), (96, 20, 40), (48, 48, 48)])
@pytest.mark.parametrize("spectrum", sorted(SPECTRA))
def test_clustered_spectra(spectrum, n):
    import paper_2401_04189_gb300 as P
    rng = np.random.default_rng(len(spectrum) * 1000 + n[0])
    s = np.sqrt(SPECTRA[spectrum])
    Q = [np.linalg.qr(rng.standard_normal((k, len(s))))[0] for k in n]
    rho = np.einsum("k,ak,bk,ck->abc", s, *Q)[None].astype(np.float32)
    one = np.ones((1, *n), dtype=np.float32)
    xs, ws = zip(*[W.uniform_grid(k, 3.0) for k in n])
    theta = np.array([4.0e4])
    sys_ = W.System("clusters", list(xs), list(ws), [q[:, :10].copy() for q in Q], theta, np.sqrt(theta), one, 0.0)
    ref = O.exchange_apply_sthosvd(one, O.Setup.from_system(sys_), (10, 10, 10), psi_tgt=rho)
    ctx = P.Context.from_system(sys_, precision="fp32")
    got = P.tx_exchange_apply_sthosvd(ctx, to_gpu(one), to_gpu(rho)).cpu().numpy()
    ctx.check_device_error()
    K = n[0] * n[1] * n[2] / min(n)
    assert rel(got, ref) < 3 * K * 2.0 ** -24
