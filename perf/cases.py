"""Timed cases of the library's calls on matrix-completion SDPs (eq. matcomp_sdp).

Each case is one call, or one short sequence of calls, that a program makes with a
problem it has set up: the Hessian matvec, the preconditioner's build and apply, a PCG
solve, one interior-point step from a given iterate, the first iterations of a batched
solve.  Shapes follow the workloads of the repository: 20 x 20 (the smallest), the batched
range p, q in [50, 400] with r in 1..4 and m = min(pq/2, 3 r (p+q) ln(p+q)), the paper's
500 x 500, 2000 x 2000 and the Fig. 1 shapes up to n = 5024.
"""
import math

import numpy as np
import torch

from paper_1703_10973_gb300 import SDPBatch, SDPProblem, default_params

F64 = torch.float64


def _m_rule(p, q, r):
    """Observation count of the batched and served workloads."""
    return int(min(p * q // 2, math.ceil(3.0 * r * (p + q) * math.log(p + q))))


def listed():
    return [
        # the Hessian product of a solver that drives its own iteration, tiny order: latency and launches
        dict(name="matvec_tiny", kind="matvec", p=20, q=20, r=1, m=200, prec="fp64"),
        # the same at a batched instance's shape: odd sides, dense samples (n = 565)
        dict(name="matvec_mid", kind="matvec", p=375, q=190, r=4, m=_m_rule(375, 190, 4), prec="fp64"),
        # the mixed form's product (float W_s split from the top eigenpairs)
        dict(name="matvec_mid_fp32", kind="matvec", p=331, q=262, r=3, m=_m_rule(331, 262, 3), prec="fp32"),
        # 2000 x 2000, sparse samples: the largest single instance that is solved to the end
        dict(name="matvec_large", kind="matvec", p=2000, q=2000, r=3, m=60000, prec="fp64"),
        # the largest shape of Fig. 1 (m = 0.025 n^2) in the lowest precision
        dict(name="matvec_max_bf16", kind="matvec", p=2512, q=2512, r=1, m=631014, prec="bf16"),
        # Algorithm 1 steps 1-2 for a new scaling matrix and one apply, batched shape
        dict(name="precond_mid", kind="precond", p=375, q=190, r=4, m=_m_rule(375, 190, 4), prec="fp64"),
        # one Newton system by PCG, Fig. 2 shape
        dict(name="pcg_1000", kind="pcg", p=500, q=500, r=4, m=20000, prec="fp64"),
        # one interior-point iteration from a mid-solve iterate: the smallest, ...
        dict(name="step_tiny", kind="step", p=20, q=20, r=1, m=200, prec="fp64"),
        # ... a batched shape, ...
        dict(name="step_mid", kind="step", p=375, q=190, r=4, m=_m_rule(375, 190, 4), prec="fp64"),
        # ... the same in the mixed form, other sizes, ...
        dict(name="step_mid_fp32", kind="step", p=400, q=311, r=2, m=_m_rule(400, 311, 2), prec="fp32"),
        # ... and a Fig. 1 shape
        dict(name="step_2000", kind="step", p=1000, q=1000, r=1, m=50000, prec="fp64"),
        # the headline workload's form: a batch of uneven instances advanced together from the start point
        dict(name="batch_4", kind="batch", p=397, q=131, r=2, m=_m_rule(397, 131, 2), prec="fp32", count=4, iters=3),
    ]


def draw(rng):
    kind = rng.choice(["matvec", "matvec", "precond", "pcg", "step", "step", "batch"])
    prec = rng.choice(["fp64", "fp64", "fp32", "bf16"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "matvec":
        p, q = size(20, 2512), size(20, 2512)
    elif kind == "precond":
        p, q = size(20, 1000), size(20, 1000)
    elif kind == "pcg":
        p, q = size(20, 500), size(20, 500)
    elif kind == "step":
        p, q = size(20, 1000), size(20, 1000)
    else:
        p, q = rng.randint(50, 400), rng.randint(50, 400)
    r = rng.randint(1, 4)
    m = min(_m_rule(p, q, r), 60000 if kind in ("matvec", "step") else 20000)
    if kind in ("precond", "step") and p + q > 1000:
        r, m = 1, min(m, 25 * (p + q))   # Fig. 1 shapes
    c = dict(kind=kind, p=p, q=q, r=r, m=m, prec=prec if kind != "precond" else "fp64")
    if kind == "batch":
        c.update(prec=rng.choice(["fp64", "fp32"]), count=rng.randint(2, 5), iters=rng.randint(1, 3))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
class _Data:
    """One matrix-completion SDP in triplet form (host arrays) with its planted factors."""

    def __init__(self, p, q, r, m, seed):
        rng = np.random.default_rng(seed)
        G1, G2 = rng.standard_normal((p, r)), rng.standard_normal((q, r))
        omega = np.sort(rng.choice(p * q, size=m, replace=False))
        self.rows, self.cols = (omega // q).astype(np.int32), (omega % q).astype(np.int32)
        self.p, self.q, self.n, self.m, self.k = p, q, p + q, m, r
        self.b = np.einsum("ij,ij->i", G1[self.rows], G2[self.cols])
        d = np.arange(self.n, dtype=np.int32)
        self.Ci, self.Cj, self.Cv = d, d, np.full(self.n, 0.5)
        self.Ak, self.Ai = np.arange(m, dtype=np.int32), self.rows
        self.Aj, self.Av = (self.cols + p).astype(np.int32), np.full(m, 0.5)
        # thin SVD of the planted matrix M = G1 G2^T = U diag(s) V^T
        Q1, R1 = np.linalg.qr(G1)
        Q2, R2 = np.linalg.qr(G2)
        u, s, vt = np.linalg.svd(R1 @ R2.T)
        self.U, self.s, self.V = Q1 @ u, s, Q2 @ vt.T


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _spread(n, lo, hi, g):
    """Random symmetric positive definite matrix with eigenvalues log-uniform in [lo, hi]:
    a diagonal turned by three Householder reflections."""
    D = torch.diag(torch.exp(torch.rand(n, generator=g, device="cuda", dtype=F64) * math.log(hi / lo) + math.log(lo)))
    for _ in range(3):
        h = torch.randn(n, generator=g, device="cuda", dtype=F64)
        h /= h.norm()
        D = D - 2.0 * torch.outer(h, h @ D)
        D = D - 2.0 * torch.outer(D @ h, h)
    return (D + D.T) / 2


def _scaling(d, seed):
    """A scaling matrix as it is in mid-solve: a bulk in [0.5, 2.5] and r large eigenvalues."""
    g = _gen(seed)
    W = _spread(d.n, 0.5, 2.5, g)
    v = torch.from_numpy(np.concatenate([d.U, d.V]) / math.sqrt(2.0)).cuda()
    lam = 20.0 + 80.0 * torch.sort(torch.rand(d.k, generator=g, device="cuda", dtype=F64)).values
    return W + (v * lam) @ v.T


def _iterate(d, seed):
    """A mid-solve iterate (X, y, S): X = the planted optimum's part + a bulk of order mu, y near
    zero, S = mu L^{-T} E L^{-1} (X = L L^T) with the eigenvalues of E spread over [0.4, 2.5], so
    that X S has the spread of an iterate off the central path."""
    g = _gen(seed)
    mu = 0.3
    v = torch.from_numpy(np.concatenate([d.U, d.V])).cuda()
    X = (v * torch.from_numpy(d.s).cuda() * 0.8) @ v.T + _spread(d.n, 0.7, 1.4, g)
    X = (X + X.T) / 2
    L = torch.linalg.cholesky(X)
    E = _spread(d.n, 0.4 * mu, 2.5 * mu, g)
    T = torch.linalg.solve_triangular(L.T.contiguous(), E, upper=True)
    S = torch.linalg.solve_triangular(L.T.contiguous(), T.T.contiguous(), upper=True)
    S = (S + S.T) / 2
    y = 0.01 * torch.randn(d.m, generator=g, device="cuda", dtype=F64)
    return X, y, S


def _vec(m, seed):
    return torch.randn(m, generator=_gen(seed), device="cuda", dtype=F64)


def _instances(case, seed):
    """The uneven instances of a batch: the case's shape, then smaller ones."""
    out = []
    for i in range(case["count"]):
        f = 1.0 - 0.17 * i
        p, q, r = max(int(case["p"] * f), 20), max(int(case["q"] * f), 20), 1 + (case["r"] + i - 1) % 4
        out.append((p, q, r, case["m"] if i == 0 else _m_rule(p, q, r), seed * 16 + i))
    return out


def prepare(case, seed):
    kind, prec = case["kind"], case["prec"]
    st = dict(kind=kind, prec=prec)
    if kind == "batch":
        prm = default_params(prec=prec, ipm_maxit=case["iters"])
        st["streams"] = [torch.cuda.Stream() for _ in range(case["count"] + 1)]   # one per problem, and the batch's
        st["problems"] = [SDPProblem.from_data(_Data(*s), params=prm, stream=t.cuda_stream)
                          for s, t in zip(_instances(case, seed), st["streams"])]
        st["batch"] = SDPBatch(st["problems"], stream=st["streams"][-1].cuda_stream)
        return st
    d = _Data(case["p"], case["q"], case["r"], case["m"], seed)
    prob = SDPProblem.from_data(d, params=default_params(prec=prec))
    st["prob"] = prob
    if kind == "step":
        st["iterate"] = [t.cpu().numpy() for t in _iterate(d, seed)]
        return st
    W = _scaling(d, seed)
    prob.set_W(W)
    st["v"] = _vec(d.m, seed + 1)
    st["out"] = torch.empty_like(st["v"])
    if kind == "precond":
        st["W"] = W
    elif kind == "pcg" or prec != "fp64":
        prob.precond_build()   # what the PCG, or the split of a reduced-precision product, starts from
    return st


def run(state):
    kind, prec = state["kind"], state["prec"]
    if kind == "batch":
        for prob in state["problems"]:
            prob.reset()
        state["batch"].solve(allow_maxit=True)
        return [list(prob.get_solution()) for prob in state["problems"]]
    prob = state["prob"]
    if kind == "matvec":
        return prob.hessian_matvec(state["v"], out=state["out"], prec=prec)
    if kind == "precond":
        prob.set_W(state["W"])
        prob.precond_build()
        return {"z": prob.precond_apply(state["v"], out=state["out"]), "tau": prob.precond_info()[0]}
    if kind == "pcg":
        return prob.pcg_solve(state["v"], rtol=1e-10, maxit=1000, prec=prec, out=state["out"])[0]
    X, y, S = state["iterate"]
    prob.set_state(X, y, S)
    prob.ipm_step()
    tau = prob.precond_info()[0]
    X1, y1, S1 = prob.get_solution()
    return {"W": prob.get_W(), "tau": tau, "X": X1, "y": y1, "S": S1}


def work(case):
    """Bytes: the operands read once and the results written once.  Flops, in FP64 terms:
    matvec: T = W V on the pattern and one length-n dot per constraint; preconditioner: the top
    eigenpairs by a few products with W and the core's factorisation; Newton system: a matvec and a
    preconditioner apply per PCG iteration, 20 of them; step: two Cholesky factors, their inverses,
    the scaling (five products) and two directions (three products each, 20 matvecs)."""
    def one(kind, p, q, r, m, prec):
        n = p + q
        ws = {"fp64": 8, "fp32": 4, "bf16": 2}[prec]
        mv = 2.0 * (2 * m) * n + 2.0 * m * n
        core = (min(p, q) * r) ** 3 / 3.0
        if kind == "matvec":
            return ws * n * n + 16.0 * m + 12.0 * 2 * m, mv
        if kind == "precond":
            return 8.0 * n * n + 16.0 * m, 2.0 * n * n * 3 * r + core
        if kind == "pcg":
            return 8.0 * n * n + 16.0 * m, 20 * mv
        return 5 * 8.0 * n * n + 16.0 * m, n ** 3 * (2 / 3.0 + 2 / 3.0 + 10.0 + 12.0) + core + 40 * mv

    if case["kind"] == "batch":
        parts = [one("step", p, q, r, m, case["prec"]) for p, q, r, m, _ in _instances(case, 0)]
        return {"bytes": sum(b for b, _ in parts), "flops": case["iters"] * sum(f for _, f in parts)}
    b, f = one(case["kind"], case["p"], case["q"], case["r"], case["m"], case["prec"])
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same results in 64 bits by plain torch
# ---------------------------------------------------------------------------
def _hess(d, W, v):
    """A(W (sum v_i A_i) W)"""
    rows, cols = torch.from_numpy(d.rows).long().cuda(), torch.from_numpy(d.cols).long().cuda() + d.p
    V = torch.zeros(d.n, d.n, dtype=F64, device="cuda")
    V[rows, cols] = 0.5 * v
    V[cols, rows] = 0.5 * v
    return (W @ (V @ W))[rows, cols]


def _eigh(A):
    w, Q = np.linalg.eigh(A.cpu().numpy())
    return torch.from_numpy(w).cuda(), torch.from_numpy(Q).cuda()


def _precond_solve(d, W, r):
    """z = Hhat^{-1} r with Hhat = A^T (tau^2 I + 2 tau U U^T kron I) A (eq. sparse_prec)."""
    n, m, k = d.n, d.m, min(d.k, d.n - 1)
    w, Q = _eigh(W)
    tau = w[0]
    U = Q[:, n - k:] * torch.sqrt(w[n - k:] - tau)
    rows, cols = torch.from_numpy(d.rows).long().cuda(), torch.from_numpy(d.cols).long().cuda() + d.p
    UU = torch.zeros(m, n, k, dtype=F64, device="cuda")   # row i: A_i . (sqrt(2 tau) e_x u_l^T)
    i = torch.arange(m, device="cuda")
    UU[i, rows] = 0.5 * torch.sqrt(2 * tau) * U[cols]
    UU[i, cols] = 0.5 * torch.sqrt(2 * tau) * U[rows]
    UU = UU.reshape(m, n * k)
    core = 2.0 * UU.T @ UU + tau ** 2 * torch.eye(n * k, dtype=F64, device="cuda")   # G = A^T A = I / 2
    L = torch.linalg.cholesky(core)
    s = torch.cholesky_solve((UU.T @ (2.0 * r))[:, None], L)[:, 0]
    return 2.0 / tau ** 2 * (r - UU @ s), tau


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None
    d = _Data(case["p"], case["q"], case["r"], case["m"], seed)
    if kind == "step":
        X, _, S = _iterate(d, seed)
        w, Q = _eigh(X)
        Xh = (Q * torch.sqrt(w)) @ Q.T
        w2, Q2 = _eigh((lambda M: (M + M.T) / 2)(Xh @ S @ Xh))
        W = Xh @ ((Q2 / torch.sqrt(w2)) @ Q2.T) @ Xh
        W = (W + W.T) / 2
        return {"W": W, "tau": float(np.linalg.eigvalsh(W.cpu().numpy())[0]), "X": None, "y": None, "S": None}
    W, v = _scaling(d, seed), _vec(d.m, seed + 1)
    if kind == "matvec":
        return _hess(d, W, v)
    if kind == "precond":
        if d.m * d.n * d.k > 1.5e9:
            return None
        z, tau = _precond_solve(d, W, v)
        return {"z": z, "tau": float(tau)}
    if d.m > 20000:
        return None
    r, c = torch.from_numpy(d.rows).long().cuda(), torch.from_numpy(d.cols).long().cuda() + d.p
    H = 0.5 * (W[r][:, r] * W[c][:, c] + W[r][:, c] * W[c][:, r])
    return torch.cholesky_solve(v[:, None], torch.linalg.cholesky(H))[:, 0]
