"""float32 kernels at the edges of their tiles, against the oracle: rows that do not fill a CTA,
several planes per CTA and several y tiles per plane, every width class of phi's columns, odd
sizes (scalar accesses), ranks above one 64-deep part, and GEMM tiles with one row or column.
Tolerances are those of the float32 parity tests."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from _helpers import E_TOL, assert_close, to_gpu

pytestmark = pytest.mark.gpu

SHAPES = [
    ((2, 3, 5), (1, 2, 3)),            # smallest: one fragment of rows, scalar columns
    ((7, 9, 17), (7, 9, 8)),           # full ranks, two column units
    ((33, 4, 130), (11, 3, 40)),       # many planes per CTA, nine units
    ((5, 150, 46), (4, 40, 21)),       # two y tiles of the projection, half a unit
    ((3, 300, 20), (2, 17, 13)),       # more rows than any CTA holds
    ((9, 21, 256), (5, 20, 33)),       # the widest phi
    ((4, 75, 78), (3, 70, 66)),        # ranks above one part
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2401_04189_gb300 import build
    build.build()


def _system(n, r, T=3, n_orb=3, seed=5):
    rng = np.random.default_rng(seed)
    xs, ws = zip(*[W.uniform_grid(k, 2.0) for k in n])
    psi = rng.standard_normal((n_orb, *n)).astype(np.float32)
    U = [np.linalg.qr(rng.standard_normal((k, q)))[0] for k, q in zip(n, r)]
    return W.System("edges", list(xs), list(ws), U, np.array([0.02, 0.9, 11.0][:T]), np.array([0.5, 0.8, 1.7][:T]), psi, 0.0)


@pytest.mark.parametrize("n,r", SHAPES)
def test_apply_energy_and_vjp(n, r):
    import torch
    import paper_2401_04189_gb300 as P
    s = _system(n, r)
    S = O.Setup.from_system(s)
    ctx = P.Context.from_system(s, precision="fp32")
    occ = to_gpu(s.psi)
    ref = O.exchange_apply(s.psi, S)
    got, e = P.tx_exchange_apply_energy(ctx, occ)
    assert_close(got.cpu().numpy(), ref, "fp32", "edges")
    ref_e = O.exchange_energy(s.psi, S, W=ref)
    scale = 0.5 * sum(np.sum(np.abs(a * b) * np.einsum("i,j,k->ijk", *s.w)) for a, b in zip(s.psi.astype(np.float64), ref))
    assert abs(float(e.item()) - ref_e) < E_TOL["fp32"] * scale
    rng = np.random.default_rng(1)
    tgt, cot = rng.standard_normal((2, 2, *n)).astype(np.float32)
    ro, rt = O.exchange_apply_vjp(s.psi, tgt, cot, S)
    go, gt = P.tx_exchange_apply_vjp(ctx, occ, to_gpu(tgt), to_gpu(cot))
    assert_close(go.cpu().numpy(), ro, "fp32", "edges-vjp-occ", scale=5)
    assert_close(gt.cpu().numpy(), rt, "fp32", "edges-vjp-tgt", scale=5)
    gal = P.tx_exchange_apply_galerkin(ctx, occ)
    assert_close(gal.cpu().numpy(), O.exchange_apply_galerkin(s.psi, S), "fp32", "edges-galerkin", scale=5)
    torch.cuda.synchronize()


@pytest.mark.parametrize("n,r", [((5, 9, 70), (3, 4, 6)), ((67, 6, 5), (5, 3, 3)), ((2, 3, 4), (2, 3, 4))])
def test_per_pair_bases_on_long_and_short_modes(n, r):
    """Eigenproblems with more rotations per round than the CTA has warps, odd sizes and the smallest;
    float32 eigenvectors are orthogonal to about 1e-6 (the bound of the per-pair parity test)."""
    import paper_2401_04189_gb300 as P
    rng = np.random.default_rng(3)
    s = _system(n, r)
    # smooth densities (decaying singular values), as the truncation needs a gap
    x, y, z = np.meshgrid(*s.x, indexing="ij")
    s.psi = np.stack([np.exp(-a * (x ** 2 + 1.3 * y ** 2 + 0.7 * z ** 2) + 0.2 * x * y)
                      for a in rng.uniform(0.3, 1.0, 3)]).astype(np.float32)
    ctx = P.Context.from_system(s, precision="fp32")
    got = P.tx_exchange_apply_sthosvd(ctx, to_gpu(s.psi)).cpu().numpy()
    ref = O.exchange_apply_sthosvd(s.psi, O.Setup.from_system(s), r)
    assert np.linalg.norm(got - ref) < 2e-5 * np.linalg.norm(ref)
