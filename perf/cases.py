"""What is timed: the work that a user of this library has it do, through its Python entry points.

A case is a dict of plain values.  Its "kind" names the entry point:

  apply     tx_exchange_apply: K psi for a block of orbitals (the call of every SCF step)
  vjp       exchange_apply under autograd, forward and backward
  batch     a BatchPlan over uneven systems, replayed as one graph
  galerkin  tx_exchange_apply_galerkin (two-sided projection)
  sthosvd   tx_exchange_apply_sthosvd (a Tucker basis of its own for every pair)
  ace       tx_ace_apply (the compressed operator, applied many times per SCF step)
  transfer  Transfer.s_to_u and Transfer.u_to_s (finite-element mesh and grid)

Orbitals are sums of s-type Gaussians on the atoms of a cluster, orthonormalised in the
quadrature weights; the Tucker basis is the HOSVD of the total density and 1/r is a sinc-rule sum
of Gaussians, as in the repository's own workloads.  Sizes are those of the repository's workloads
(small, Pt-shaped, TiO2-shaped, differentiation, uneven batch) with fewer orbitals where the whole
block takes long: a pair costs the same however many there are.
"""
import itertools
import math

import numpy as np
import torch

import paper_2401_04189_gb300 as P

DEV = "cuda"


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------
def _apply(name, prec, n, r, T, half, occ, tgt, block):
    n, r = (n,) * 3 if isinstance(n, int) else n, (r,) * 3 if isinstance(r, int) else r
    return dict(name=name, kind="apply", prec=prec, n1=n[0], n2=n[1], n3=n[2], r1=r[0], r2=r[1], r3=r[2], T=T,
                half=float(half), occ=occ, tgt=tgt, targets=block)


def listed():
    return [
        # a molecule: 4 orbitals on a small grid, where launches and latency are the whole time
        _apply("apply_small_bf16", "bf16", 32, 16, 30, 8, 4, 4, "all"),
        # the Pt cluster: every orbital a target, one apply per SCF step in the fast precision
        _apply("apply_pt_bf16", "bf16", 96, 40, 40, 12, 64, 64, "all"),
        # one share of the TiO2 cluster's pairs: the largest grid, rank and term count
        _apply("apply_tio2_bf16", "bf16", 160, 64, 45, 16, 32, 8, "slice"),
        # an anisotropic box with a grid and ranks that are no multiples of any tile, targets that
        # are other orbitals than the occupied ones (virtual orbitals, trial vectors)
        _apply("apply_ragged_tf32", "tf32", (75, 90, 100), (20, 33, 41), 37, 11, 20, 12, "other"),
        # the Pt cluster where 1e-6 is asked for (final SCF steps, energy differences)
        _apply("apply_pt_tf32x3", "tf32x3", 96, 40, 40, 12, 24, 24, "all"),
        # the float32 form, the one that every other is checked against and the one for small systems
        _apply("apply_pt_fp32", "fp32", 96, 40, 40, 12, 16, 16, "all"),
        # differentiating through K: the forward and both gradients, at the split precision
        dict(name="vjp_diff_tf32x3", kind="vjp", prec="tf32x3", n1=64, n2=64, n3=64, r1=32, r2=32, r3=32, T=35,
             half=10.0, occ=16, tgt=8),
        # screening many small systems at once: six uneven ones, one captured graph
        dict(name="batch_uneven_bf16", kind="batch", prec="bf16",
             systems="96,37,36,10;64,25,33,10;112,43,38,8;48,20,30,12;80,48,40,10;64,31,35,16"),
        # the symmetric form of the operator at truncated rank
        dict(name="galerkin_diff", kind="galerkin", prec="fp32", n1=64, n2=64, n3=64, r1=32, r2=32, r3=32, T=35,
             half=10.0, occ=16, tgt=16, targets="all"),
        # the paper's own decomposition, a basis for every pair
        dict(name="sthosvd_48", kind="sthosvd", prec="fp32", n1=48, n2=48, n3=48, r1=20, r2=20, r3=20, T=30, half=6.0,
             occ=8, tgt=8, targets="all"),
        # V_ACE psi for a block of trial vectors: what the eigensolver calls inside an SCF step
        dict(name="ace_pt", kind="ace", prec="fp32", n1=96, n2=96, n3=96, half=12.0, occ=64, tgt=64),
        # orbitals to the grid and back: second-order mesh cells refined at the atoms, third-order grid cells
        dict(name="transfer_tio2", kind="transfer", n1=160, n2=160, n3=160, half=16.0, base=9, order_u=2, order_s=3,
             orbitals=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply"] * 6 + ["vjp", "batch", "galerkin", "sthosvd", "ace", "transfer"])
    if kind == "apply":
        prec = rng.choice(["bf16", "bf16", "tf32", "tf32x3", "tf32x3", "bf16x3", "fp32", "fp32"])
        top = {"bf16": 160, "tf32": 128, "tf32x3": 128, "bf16x3": 96, "fp32": 120}[prec]
        n = [_log_int(rng, 24, top) for _ in range(3)]
        n[2] = max(24, 4 * (n[2] // 4))                       # 16-byte grid rows (the tensor-core precisions ask for them)
        r = [min(m // 2, rng.randint(12, 64)) for m in n]
        T = rng.randint(25, 45)
        budget = {"bf16": 6e12, "tf32": 3e12, "tf32x3": 5e11, "bf16x3": 5e11, "fp32": 2e11}[prec]
        targets = rng.choice(["all", "slice", "other"])
        cost = _pair_flops(n, r, T)
        pairs = max(1, min(1200, int(budget * math.exp(rng.uniform(math.log(0.02), 0.0)) / cost)))
        occ = max(2, min(40, int(math.sqrt(2 * pairs))))
        tgt = occ if targets == "all" else max(1, min(occ - 1, rng.randint(1, occ)))
        return dict(kind="apply", prec=prec, n1=n[0], n2=n[1], n3=n[2], r1=r[0], r2=r[1], r3=r[2], T=T,
                    half=max(n) / 8.0, occ=occ, tgt=tgt, targets=targets)
    if kind == "vjp":
        n = [_log_int(rng, 28, 72) for _ in range(3)]
        n[2] = max(28, 4 * (n[2] // 4))
        r = [min(m // 2, rng.randint(12, 32)) for m in n]
        occ = rng.randint(2, 10)
        return dict(kind="vjp", prec=rng.choice(["tf32x3", "fp32"]), n1=n[0], n2=n[1], n3=n[2], r1=r[0], r2=r[1],
                    r3=r[2], T=rng.randint(25, 40), half=max(n) / 6.4, occ=occ, tgt=rng.randint(1, occ))
    if kind == "batch":
        sysn = [",".join(str(v) for v in (rng.choice([48, 64, 80, 96, 112]), rng.randint(20, 48), rng.randint(30, 40),
                                          rng.randint(4, 10))) for _ in range(rng.randint(2, 6))]
        return dict(kind="batch", prec=rng.choice(["bf16", "bf16", "tf32"]), systems=";".join(sysn))
    if kind in ("galerkin", "sthosvd"):
        big = kind == "galerkin"
        n = [_log_int(rng, 24, 80 if big else 50) for _ in range(3)]
        r = [min(m // 2, rng.randint(10, 36 if big else 22)) for m in n]
        occ = rng.randint(3, 14 if big else 6)
        targets = rng.choice(["all", "other"])
        return dict(kind=kind, prec="fp32", n1=n[0], n2=n[1], n3=n[2], r1=r[0], r2=r[1], r3=r[2], T=rng.randint(20, 36),
                    half=max(n) / 8.0, occ=occ, tgt=occ if targets == "all" else rng.randint(1, occ), targets=targets)
    if kind == "ace":
        n = [_log_int(rng, 32, 110) for _ in range(3)]
        return dict(kind="ace", prec="fp32", n1=n[0], n2=n[1], n3=n[2], half=max(n) / 8.0, occ=_log_int(rng, 3, 80),
                    tgt=_log_int(rng, 1, 80))
    order_s = rng.choice([1, 2, 3])
    n = [order_s * rng.randint(30 // order_s, 130 // order_s) + 1 for _ in range(3)]
    return dict(kind="transfer", n1=n[0], n2=n[1], n3=n[2], half=max(n) / 10.0, base=rng.randint(5, 10),
                order_u=rng.choice([1, 2, 3]), order_s=order_s, orbitals=_log_int(rng, 3, 64))


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _dims(case):
    return [case["n1"], case["n2"], case["n3"]]


def _ranks(case):
    return [case["r1"], case["r2"], case["r3"]]


def _grid(n, half):
    xs = [np.linspace(-half, half, k) for k in n]
    ws = []
    for k in n:
        w = np.full(k, 2.0 * half / (k - 1))
        w[0] = w[-1] = 0.5 * w[1]
        ws.append(w)
    return xs, ws


def _gaussian_sum(n, half, T):
    """1/r = (2/sqrt(pi)) int exp(-r^2 e^{2s} + s) ds by the trapezoid rule over the s that matter
    between the grid spacing and the box diagonal; the rest of the rule below joins the first term."""
    h = min(2.0 * half / (k - 1) for k in n)
    s_hi, s_lo = -math.log(h) + 1.15, -math.log(math.sqrt(3.0) * 2.0 * half) - 5.0
    d = (s_hi - s_lo) / (T - 1)
    s = s_lo + d * np.arange(T)
    c = 2.0 / math.sqrt(math.pi) * d
    mu = c * np.exp(s)
    mu[0] += c * math.exp(s[0]) * math.exp(-d) / (1.0 - math.exp(-d))
    return np.exp(2.0 * s), mu


def _orbitals(xs, ws, half, count, rng, atoms=24, per_orbital=6, per_atom=2):
    """Loewdin-orthonormal sums of Gaussians (exponents U[0.2, 3], coefficients N(0, 1)) on atoms of a
    cluster that fills the middle of the box: float32 [count, n1, n2, n3] on the device."""
    f64 = dict(dtype=torch.float64, device=DEV)
    centres = rng.uniform(-0.45 * half, 0.45 * half, size=(atoms, 3))
    K = per_orbital * per_atom
    x = [torch.tensor(v, **f64) for v in xs]
    psi = torch.empty((count, len(xs[0]), len(xs[1]), len(xs[2])), **f64)
    for i in range(count):
        cen = np.repeat(centres[rng.choice(atoms, size=per_orbital, replace=False)], per_atom, axis=0)
        a = torch.tensor(rng.uniform(0.2, 3.0, size=K), **f64)[:, None]
        c = torch.tensor(rng.standard_normal(K), **f64)[:, None]
        e = [torch.exp(-a * (x[d][None, :] - torch.tensor(cen[:, d], **f64)[:, None]) ** 2) for d in range(3)]
        psi[i] = ((c * e[0])[:, :, None] * e[1][:, None, :]).reshape(K, -1).T.matmul(e[2]).reshape(psi.shape[1:])
    w = [torch.tensor(v, **f64) for v in ws]
    flat = psi.reshape(count, -1)
    S = (flat * (w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]).reshape(1, -1)) @ flat.T
    ev, V = torch.linalg.eigh(S.cpu())
    X = ((V * ev.clamp(min=1e-8 * float(ev.max())) ** -0.5) @ V.T).to(DEV)
    return (X @ flat).reshape(psi.shape).to(torch.float32)


def _basis(psi, r):
    rho = (psi.to(torch.float64) ** 2).sum(0)
    U = []
    for d in range(3):
        M = torch.movedim(rho, d, 0).reshape(rho.shape[d], -1)
        _, V = torch.linalg.eigh((M @ M.T).cpu())
        U.append(np.ascontiguousarray(V.flip(1)[:, :r[d]].numpy()))
    return U


def _system(case, seed):
    n, half = _dims(case), case["half"]
    rng = np.random.default_rng(seed)
    xs, ws = _grid(n, half)
    theta, mu = _gaussian_sum(n, half, case["T"])
    other = case.get("targets", "other") == "other"
    psi = _orbitals(xs, ws, half, case["occ"] + (case["tgt"] if other else 0), rng)
    occ = psi[:case["occ"]]
    U = _basis(occ, _ranks(case))
    tgt = psi[case["occ"]:].contiguous() if other else (occ[:case["tgt"]] if case["targets"] == "slice" else None)
    return dict(xs=xs, ws=ws, U=U, theta=theta, mu=mu, occ=occ.contiguous() if other else occ, tgt=tgt)


def _batch_systems(case, seed):
    for k, text in enumerate(case["systems"].split(";")):
        n, r, T, occ = (int(v) for v in text.split(","))
        yield _system(dict(n1=n, n2=n, n3=n, r1=r, r2=r, r3=r, T=T, half=n / 8.0, occ=occ, tgt=occ, targets="all"),
                      1000 * seed + k)


def _mesh(half, base, order):
    """base^3 cubic cells, those near one of five atoms split into eight (hanging nodes stay): nodes [., 3] and
    cells [., (order + 1)^3].  The mesh belongs to the case, the orbitals on it to the seed."""
    atoms = np.random.default_rng(base).uniform(-0.6 * half, 0.6 * half, size=(5, 3))
    h = 2.0 * half / base
    lo = -half + h * np.stack(np.meshgrid(*[np.arange(base)] * 3, indexing="ij"), -1).reshape(-1, 3)
    near = np.min(np.linalg.norm(lo[:, None, :] + 0.5 * h - atoms[None], axis=2), axis=1) < 1.2 * h
    kids = np.array(list(itertools.product((0, 1), repeat=3)))
    lo = np.concatenate([lo[~near], (lo[near][:, None, :] + 0.5 * h * kids[None]).reshape(-1, 3)])
    width = np.concatenate([np.full((~near).sum(), h), np.full(8 * near.sum(), 0.5 * h)])
    q = np.stack(np.meshgrid(*[np.arange(order + 1) / order] * 3, indexing="ij"), -1).reshape(-1, 3)
    pts = lo[:, None, :] + width[:, None, None] * q[None]
    key = np.round((pts.reshape(-1, 3) + half) / (1e-7 * half)).astype(np.int64)
    _, first, conn = np.unique(key, axis=0, return_index=True, return_inverse=True)
    return pts.reshape(-1, 3)[first], conn.reshape(len(lo), -1).astype(np.int32)


def _context(s, prec):
    ctx = P.Context(s["xs"], s["ws"], s["U"], s["theta"], s["mu"], precision=prec)
    ctx.set_workspace_limit(16 << 30)      # as the benchmark does: the card has 280 GB
    return ctx


def _ace_inputs(case, seed):
    rng = np.random.default_rng(seed)
    xs, ws = _grid(_dims(case), case["half"])
    xi = _orbitals(xs, ws, case["half"], case["occ"], rng)
    scale = torch.tensor(rng.uniform(0.3, 1.2, size=case["occ"]), dtype=torch.float32, device=DEV)
    return xs, ws, xi * scale[:, None, None, None], _orbitals(xs, ws, case["half"], case["tgt"], rng)


def _transfer_inputs(case, seed):
    xs, ws = _grid(_dims(case), case["half"])
    X, conn = _mesh(case["half"], case["base"], case["order_u"])
    gen = torch.Generator(device=DEV).manual_seed(seed)
    psi_s = torch.randn((case["orbitals"], *_dims(case)), generator=gen, device=DEV)
    psi_u = torch.randn((X.shape[0], case["orbitals"]), generator=gen, device=DEV)
    return xs, ws, X, conn, psi_s, psi_u


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        systems = list(_batch_systems(case, seed))
        ctxs = [_context(s, case["prec"]) for s in systems]
        plan = P.BatchPlan([dict(ctx=c, psi_occ=s["occ"]) for c, s in zip(ctxs, systems)])
        plan.capture(torch.cuda.Stream())
        return dict(kind=kind, plan=plan, ctxs=ctxs)
    if kind == "ace":
        xs, ws, xi, psi = _ace_inputs(case, seed)
        eye = [np.eye(len(x))[:, :1] for x in xs]
        ctx = P.Context(xs, ws, eye, [1.0], [1.0], precision=case["prec"])
        return dict(kind=kind, ctx=ctx, xi=xi, psi=psi)
    if kind == "transfer":
        xs, ws, X, conn, psi_s, psi_u = _transfer_inputs(case, seed)
        ctx = P.Context(xs, ws, [np.eye(len(x))[:, :1] for x in xs], [1.0], [1.0], precision="fp32")
        return dict(kind=kind, ctx=ctx, tr=P.Transfer(ctx, X, conn, case["order_u"], case["order_s"]), psi_s=psi_s,
                    psi_u=psi_u)
    s = _system(case, seed)
    state = dict(kind=kind, ctx=_context(s, case["prec"]), occ=s["occ"], tgt=s["tgt"])
    if kind == "vjp":
        rng = torch.Generator(device=DEV).manual_seed(seed)
        state["cot"] = torch.randn(s["tgt"].shape, generator=rng, device=DEV)
        state["occ"].requires_grad_(True)
        state["tgt"].requires_grad_(True)
    return state


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return P.tx_exchange_apply(state["ctx"], state["occ"], state["tgt"])
    if kind == "vjp":
        W = P.exchange_apply(state["ctx"], state["occ"], state["tgt"])
        g_occ, g_tgt = torch.autograd.grad(W, (state["occ"], state["tgt"]), state["cot"])
        return W.detach(), g_occ, g_tgt
    if kind == "batch":
        state["plan"].replay()
        return state["plan"].outputs()
    if kind == "galerkin":
        return P.tx_exchange_apply_galerkin(state["ctx"], state["occ"], state["tgt"])
    if kind == "sthosvd":
        return P.tx_exchange_apply_sthosvd(state["ctx"], state["occ"], state["tgt"])
    if kind == "ace":
        return P.tx_ace_apply(state["ctx"], state["xi"], state["psi"])
    return state["tr"].s_to_u(state["psi_s"]), state["tr"].u_to_s(state["psi_u"])


# ------------------------------------------------------------------------------------------
# the work of one pass
# ------------------------------------------------------------------------------------------
def _mode_flops(n, r):
    """A core of ranks r expanded to a grid n (or projected from it), mode by mode."""
    return 2.0 * (n[0] * r[0] * r[1] * r[2] + n[0] * n[1] * r[1] * r[2] + n[0] * n[1] * n[2] * r[2])


def _pair_flops(n, r, T):
    """One projection, T expansions, the products with two orbitals: the method's own count, term by term."""
    return (T + 1) * _mode_flops(n, r) + 3.0 * n[0] * n[1] * n[2]


def _pairs(case):
    o, t = case["occ"], case["tgt"]
    return o * t - (t * (t - 1) // 2 if case.get("targets", "other") != "other" else 0)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        fl = by = 0.0
        for text in case["systems"].split(";"):
            n, r, T, occ = (int(v) for v in text.split(","))
            fl += occ * (occ + 1) // 2 * _pair_flops([n] * 3, [r] * 3, T)
            by += 8.0 * occ * n ** 3
        return dict(bytes=by, flops=fl)
    n = _dims(case)
    n3 = float(n[0] * n[1] * n[2])
    if kind == "ace":
        return dict(bytes=4.0 * n3 * (case["occ"] + 2 * case["tgt"]), flops=4.0 * n3 * case["occ"] * case["tgt"])
    if kind == "transfer":
        nu, ns = (case["order_u"] + 1) ** 3, (case["order_s"] + 1) ** 3
        nodes = float(case["base"] * case["order_u"] + 1) ** 3          # before refinement
        return dict(bytes=4.0 * case["orbitals"] * (n3 + nodes) * 2, flops=2.0 * case["orbitals"] * (n3 * nu + nodes * ns))
    pairs, r, T = _pairs(case), _ranks(case), case["T"]
    if kind == "vjp":    # the forward, the adjoint's first pass and the adjoint of every pair
        return dict(bytes=4.0 * n3 * (2 * case["occ"] + 4 * case["tgt"]), flops=3.0 * pairs * _pair_flops(n, r, T))
    out = dict(bytes=4.0 * n3 * (case["occ"] + case["tgt"] * (2 if case["targets"] == "other" else 1)),
               flops=pairs * _pair_flops(n, r, T))
    if kind == "galerkin":
        out["flops"] = pairs * (2 * _mode_flops(n, r) + T * _mode_flops(r, r) + 3.0 * n3)
    if kind == "sthosvd":
        grams = 2.0 * n3 * (n[0] + r[0]) + 2.0 * r[0] * n[1] * n[2] * (n[1] + r[1]) + 2.0 * r[0] * r[1] * n[2] * (n[2] + r[2])
        ops = 2.0 * T * sum(a * a * b for a, b in zip(n, r))
        out["flops"] = pairs * (grams + ops + T * _mode_flops(n, r) + 3.0 * n3)
    return out


# ------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------
def _f64(a):
    return torch.as_tensor(np.asarray(a) if not torch.is_tensor(a) else a).to(device=DEV, dtype=torch.float64)


class _Exact:
    """The operator of one system in float64: phi = sum_t mu_t G x_d (C_td U_d), G = rho x_d U_d^T."""

    def __init__(self, s):
        self.x, self.w, self.U = ([_f64(v) for v in s[k]] for k in ("xs", "ws", "U"))
        self.theta, self.mu = s["theta"], s["mu"]
        self.C = [[self.w[d][None, :] * torch.exp(-th * (self.x[d][:, None] - self.x[d][None, :]) ** 2)
                   for th in self.theta] for d in range(3)]
        self.A = [[c @ self.U[d] for c in self.C[d]] for d in range(3)]

    @staticmethod
    def modes(q, m):
        """q [B, a, b, c] with its three modes multiplied by m[d] [out_d, in_d]."""
        B, a, b, c = q.shape
        q = torch.matmul(m[0], q.reshape(B, a, b * c)).reshape(B * m[0].shape[0], b, c)
        q = torch.matmul(m[1], q)
        return torch.matmul(q.reshape(-1, c), m[2].T).reshape(B, m[0].shape[0], m[1].shape[0], m[2].shape[0])

    def core(self, rho):
        # the longest contraction first
        q = torch.matmul(rho.reshape(-1, rho.shape[3]), self.U[2]).reshape(*rho.shape[:3], -1)
        B, a, b, c = q.shape
        q = torch.matmul(self.U[1].T, q.reshape(B * a, b, c)).reshape(B, a, -1)
        return torch.matmul(self.U[0].T, q).reshape(B, self.U[0].shape[1], self.U[1].shape[1], c)

    def potential(self, rho):
        G, phi = self.core(rho), 0.0
        for t in range(len(self.theta)):
            phi = phi + self.mu[t] * self.modes(G, [self.A[d][t] for d in range(3)])
        return phi

    def adjoint(self, y):
        H = 0.0
        for t in range(len(self.theta)):
            q = torch.matmul(y.reshape(-1, y.shape[3]), self.A[2][t]).reshape(*y.shape[:3], -1)
            B, a, b, c = q.shape
            q = torch.matmul(self.A[1][t].T, q.reshape(B * a, b, c)).reshape(B, a, -1)
            H = H + self.mu[t] * torch.matmul(self.A[0][t].T, q).reshape(B, self.A[0][t].shape[1], -1, c)
        return self.modes(H, self.U)

    def potential_galerkin(self, rho):
        G, H = self.core(rho), 0.0
        for t in range(len(self.theta)):
            H = H + self.mu[t] * self.modes(G, [self.U[d].T @ (self.w[d][:, None] * self.A[d][t]) for d in range(3)])
        return self.modes(H, [self.U[d] / self.w[d][:, None] for d in range(3)])

    def potential_own_basis(self, rho, r):
        out = []
        for q in rho:
            n, g, U = q.shape, q, []
            for d in range(3):
                M = torch.movedim(g, d, 0).reshape(n[d], -1)
                _, V = torch.linalg.eigh((M @ M.T).cpu())
                U.append(V.flip(1)[:, :r[d]].contiguous().to(DEV))
                g = torch.movedim(torch.tensordot(U[d].T, g, dims=([1], [d])), 0, d)
            phi = 0.0
            for t in range(len(self.theta)):
                phi = phi + self.mu[t] * self.modes(g[None], [self.C[d][t] @ U[d] for d in range(3)])
            out.append(phi[0])
        return torch.stack(out)


def _exact_apply(s, case, potential, chunk=8):
    occ = _f64(s["occ"])
    other = case["targets"] == "other"
    tgt = _f64(s["tgt"]) if other else occ[:case["tgt"]]
    W = torch.zeros_like(tgt)
    pairs = [(i, j) for i in range(len(tgt)) for j in range(0 if other else i, len(occ))]
    for k in range(0, len(pairs), chunk):
        part = pairs[k:k + chunk]
        phi = potential(torch.stack([tgt[i] * occ[j] for i, j in part]))
        for f, (i, j) in zip(phi, part):
            W[i] -= occ[j] * f
            if not other and i < j < len(tgt):
                W[j] -= tgt[i] * f
    return W


def _lagrange(nodes, x):
    """[len(x), len(nodes)] values at x of the Lagrange polynomials on the nodes."""
    out = np.ones((len(x), len(nodes)))
    for k, m in itertools.permutations(range(len(nodes)), 2):
        out[:, k] *= (x - nodes[m]) / (nodes[k] - nodes[m])
    return out


def _exact_transfer(case, seed):
    xs, _, X, conn, psi_s, psi_u = _transfer_inputs(case, seed)
    n, pu, ps = _dims(case), case["order_u"], case["order_s"]
    psi_u64, psi_s64 = psi_u.double(), psi_s.double()
    # to the grid: the first cell that holds a node gives its value, so later cells do not overwrite it
    out = torch.zeros((case["orbitals"], *n), dtype=torch.float64, device=DEV)
    for c in range(len(conn) - 1, -1, -1):
        ax = [X[conn[c].reshape((pu + 1,) * 3)[tuple(slice(None) if d == e else 0 for e in range(3))], d] for d in range(3)]
        sel = []
        for d in range(3):
            tol = 1e-9 * (ax[d].max() - ax[d].min())
            sel.append((int(np.searchsorted(xs[d], ax[d].min() - tol)), int(np.searchsorted(xs[d], ax[d].max() + tol, side="right"))))
        if any(b <= a for a, b in sel):
            continue
        L = [_f64(_lagrange(ax[d], xs[d][sel[d][0]:sel[d][1]])) for d in range(3)]
        v = psi_u64[torch.as_tensor(conn[c].astype(np.int64), device=DEV)].T.reshape(-1, pu + 1, pu + 1, pu + 1)
        out[:, sel[0][0]:sel[0][1], sel[1][0]:sel[1][1], sel[2][0]:sel[2][1]] = _Exact.modes(v, L)
    # to the mesh: the element of the grid that holds a node, the lower one on a shared face
    base, L = [], []
    for d in range(3):
        starts = xs[d][::ps][:-1]
        e = np.clip(np.searchsorted(starts, X[:, d], side="left") - 1, 0, len(starts) - 1)
        base.append(torch.as_tensor(ps * e, device=DEV))
        nodes = np.stack([xs[d][ps * e + k] for k in range(ps + 1)], 1)
        v = np.ones_like(nodes)
        for k, m in itertools.permutations(range(ps + 1), 2):
            v[:, k] *= (X[:, d] - nodes[:, m]) / (nodes[:, k] - nodes[:, m])
        L.append(_f64(v))
    back = torch.zeros((len(X), case["orbitals"]), dtype=torch.float64, device=DEV)
    for a, b, c in itertools.product(range(ps + 1), repeat=3):
        back += (L[0][:, a] * L[1][:, b] * L[2][:, c])[:, None] * psi_s64[:, base[0] + a, base[1] + b, base[2] + c].T
    return back, out


def exact(case, seed):
    kind = case["kind"]
    if kind == "transfer":
        return _exact_transfer(case, seed)
    if kind == "ace":
        _, ws, xi, psi = _ace_inputs(case, seed)
        w = [_f64(v) for v in ws]
        wf = (w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]).reshape(1, -1)
        x, p = xi.double().reshape(len(xi), -1), psi.double().reshape(len(psi), -1)
        return (-((p * wf) @ x.T) @ x).reshape(psi.shape)
    if work(case)["flops"] > 1.2e13:
        return None          # more than a float64 pass does in 20 seconds
    if kind == "batch":
        return [_exact_apply(s, dict(targets="all", tgt=len(s["occ"])), _Exact(s).potential)
                for s in _batch_systems(case, seed)]
    s = _system(case, seed)
    op = _Exact(s)
    if kind == "vjp":
        occ, tgt = _f64(s["occ"]), _f64(s["tgt"])
        rng = torch.Generator(device=DEV).manual_seed(seed)
        cot = torch.randn(s["tgt"].shape, generator=rng, device=DEV).double()
        W, g_occ, g_tgt = torch.zeros_like(tgt), torch.zeros_like(occ), torch.zeros_like(tgt)
        for k in range(len(tgt)):
            phi, zeta = op.potential(tgt[k] * occ), op.adjoint(cot[k] * occ)
            W[k] = -(occ * phi).sum(0)
            g_tgt[k] = -(occ * zeta).sum(0)
            g_occ -= cot[k] * phi + tgt[k] * zeta
        return W, g_occ, g_tgt
    if kind == "galerkin":
        return _exact_apply(s, case, op.potential_galerkin)
    if kind == "sthosvd":
        return _exact_apply(s, case, lambda rho: op.potential_own_basis(rho, _ranks(case)))
    return _exact_apply(s, case, op.potential)
