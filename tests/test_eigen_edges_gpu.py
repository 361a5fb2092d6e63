"""Eigensolver pieces (bisection, inverse iteration, back-transformation) at the orders
where their blocks, warps and rescaling steps change, through the public calls.

Tolerances.  tau = lambda_min(W): bisection is exact to 2 eps |T|, the Householder
reduction backward stable to about n eps ||W||, so |tau - exact| <= 4 n eps ||W||_2.
NT scaling: W S W = X holds to about n eps times the condition numbers that enter
(Cholesky factor of X, eigenvectors, Lambda^(-1/2)), below 50 n eps kappa(X) kappa(S) here.
"""
import numpy as np
import pytest

import sdp_inputs as si
from oracle import sdp_oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10973_gb300 import _build, load
    _build.build()
    load()


def _prob(d, **kw):
    from paper_1703_10973_gb300 import SDPProblem, default_params
    return SDPProblem.from_data(d, params=default_params(**kw))


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()


def _spectrum(n, ev, seed):
    Q, _ = np.linalg.qr(np.random.default_rng(seed).standard_normal((n, n)))
    A = (Q * ev) @ Q.T
    return (A + A.T) / 2


@pytest.mark.parametrize("n", [2, 3, 15, 16, 17, 18, 31, 33, 34, 64, 129, 670, 690, 1380])
def test_tau_and_apply_at_edge_orders(n):
    p = n // 2
    d = si.mc_instance(p, n - p, 1, max(1, p * (n - p) // (2 if n < 100 else 40)), n)
    rng = np.random.default_rng(n)
    k = min(2, n - 1)
    W = _spectrum(n, np.concatenate([rng.uniform(0.5, 3.0, n - k), rng.uniform(30.0, 60.0, k)]), n + 1)
    tau_ref = np.linalg.eigvalsh(W)[0]
    with _prob(d, k=k) as prob:
        prob.set_W(_dev(W))
        prob.precond_build()
        tau, kk = prob.precond_info()
        r = si.random_vec(d.m, 2)
        z = prob.precond_apply(_dev(r)).cpu().numpy()
    assert kk == k
    assert abs(tau - tau_ref) <= 4 * n * EPS * 60.0
    if n <= 129:
        P = o.Problem.from_data(d)
        pc = o.precond_hat_build(P, W, k)
        H = o.precond_dense(P, pc)
        zref = np.linalg.solve(H, r)
        assert np.linalg.norm(z - zref) <= max(1e-12, 20 * np.linalg.cond(H) * EPS) * np.linalg.norm(zref)


def test_top_pairs_of_a_reducible_matrix():
    """Equal diagonal blocks: T falls apart, the inverse iteration works per block."""
    n, b = 48, 6
    B = _spectrum(b, np.array([0.7, 1.0, 1.3, 1.9, 2.5, 40.0]), 3)
    W = np.kron(np.eye(n // b), B)
    d = si.mc_instance(n // 2, n - n // 2, 1, 200, 5)
    with _prob(d, k=8) as prob:
        prob.set_W(_dev(W))
        prob.precond_build()
        tau, k = prob.precond_info()
        r = si.random_vec(d.m, 2)
        z = prob.precond_apply(_dev(r)).cpu().numpy()
    P = o.Problem.from_data(d)
    pc = o.precond_hat_build(P, W, 8)
    zref = np.linalg.solve(o.precond_dense(P, pc), r)
    assert k == 8 and abs(tau - 0.7) <= 4 * n * EPS * 40.0
    assert np.linalg.norm(z - zref) <= 20 * np.linalg.cond(o.precond_dense(P, pc)) * EPS * np.linalg.norm(zref)


@pytest.mark.parametrize("n", [2, 3, 16, 33, 65, 149, 297, 671])
def test_nt_scaling_at_edge_orders(n):
    d = si.unit_diag_instance(n)
    rng = np.random.default_rng(n)
    X, S = _spectrum(n, rng.uniform(0.5, 2.0, n), 1), _spectrum(n, rng.uniform(0.5, 2.0, n), 2)
    with _prob(d) as prob:
        prob.set_state(X, np.zeros(d.m), S, 0)
        prob.ipm_step()
        W = prob.get_W().cpu().numpy()
    assert np.linalg.norm(W @ S @ W - X) <= 50 * n * EPS * 16.0 * np.linalg.norm(X)


@pytest.mark.parametrize("n", [63, 64, 255, 256, 257, 519, 1025, 2047])
def test_step_length_is_close_to_the_boundary(n):
    """alpha = min(1, 0.9 / -(theta - bound)) with bound <= 1e-3 |theta| and theta - bound <=
    lambda_min(L^-1 dX L^-T) up to rounding: 0.998 of the largest step at least, never beyond it
    (both sides of the order where the whole-GPU Lanczos takes over, and of the matrix sizes of
    the resident tridiagonalisation)."""
    d = si.unit_diag_instance(n)
    rng = np.random.default_rng(n)
    q = min(n, 8)   # spectra without an n x n factorisation: I + low rank
    U, V = rng.standard_normal((n, q)) / np.sqrt(n), rng.standard_normal((n, q)) / np.sqrt(n)
    X, S = 0.7 * np.eye(n) + U @ U.T, 0.9 * np.eye(n) + V @ V.T
    with _prob(d) as prob:
        prob.set_state(X, np.zeros(d.m), S, 0)
        info = prob.ipm_step()
        X1, _, _ = prob.get_solution()
    a = info["alpha_p"]
    if a >= 1.0:
        return
    L = np.linalg.cholesky(X)
    D = np.linalg.solve(L, np.linalg.solve(L, (X1 - X) / a).T)
    amax = -1.0 / np.linalg.eigvalsh((D + D.T) / 2)[0]
    assert 0.9 * 0.998 * amax * (1 - 1e-7) <= a <= 0.9 * amax * (1 + 1e-7)


@pytest.mark.parametrize("n", [48, 606])
def test_nt_scaling_of_block_matrices(n):
    """Diagonal blocks of order 6: the tridiagonal form falls apart, every vector works on its own
    block, with one vector per CTA (48) and with eight (606)."""
    rng = np.random.default_rng(n)
    X, S = np.zeros((n, n)), np.zeros((n, n))
    for b in range(0, n, 6):   # spectra that differ from block to block
        X[b:b + 6, b:b + 6] = _spectrum(6, rng.uniform(0.5, 2.0, 6), b)
        S[b:b + 6, b:b + 6] = _spectrum(6, rng.uniform(0.5, 2.0, 6), b + 1)
    with _prob(si.unit_diag_instance(n)) as prob:
        prob.set_state(X, np.zeros(n), S, 0)
        prob.ipm_step()
        W = prob.get_W().cpu().numpy()
    assert np.linalg.norm(W @ S @ W - X) <= 50 * n * EPS * 16.0 * np.linalg.norm(X)
