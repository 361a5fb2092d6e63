"""Tridiagonalisation above order 1024: the resident form up to 2048, beyond it the one that streams the
matrix -- its results on both sides of that order, a grid barrier's wait that runs out in either, and the
step lengths, which need a factor of the iterate and the smallest eigenvalue only."""
import numpy as np
import pytest

import sdp_inputs as si

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


def _spectrum(n, ev, seed):
    """Symmetric with the eigenvalues ev: a diagonal turned by three reflections."""
    rng = np.random.default_rng(seed)
    A = np.diag(ev)
    for _ in range(3):
        h = rng.standard_normal(n)
        h /= np.linalg.norm(h)
        A -= 2.0 * np.outer(h, h @ A)
        A -= 2.0 * np.outer(A @ h, h)
    return (A + A.T) / 2


@pytest.mark.parametrize("n", [1025, 2049])
def test_tridiagonalisation_wait_runs_out(n):
    from paper_1703_10973_gb300 import SDPError, SDPProblem, _lib, default_params
    d = si.mc_instance(n // 2, n - n // 2, 1, 4 * n, n)
    with SDPProblem.from_data(d, params=default_params(wait_cycles=1)) as p:
        p.set_W(torch.eye(n, dtype=torch.float64, device="cuda"))
        with pytest.raises(SDPError) as e:
            p.precond_build()
        assert e.value.status == _lib.SDP_ERR_TIMEOUT
        assert "timeout" in p.lib.sdp_last_error(p.h).decode()


@pytest.mark.parametrize("n", [1025, 2047, 2048, 2049, 2100])
def test_top_pairs_above_order_1024(n):
    """tau: the reduction is backward stable and the bisection exact, |tau - exact| <= 4 n eps ||W||.
    Apply: z solves Hhat z = r, (Hhat z)_i = tau^2 ||A_i||^2 z_i + 2 tau <A_i, V U U^T>, V = sum z_i A_i,
    with U from the exact pairs, to 4 n eps kappa(Hhat), kappa(Hhat) <= 1 + 2 lambda_max / tau."""
    from paper_1703_10973_gb300 import SDPProblem, default_params
    rng = np.random.default_rng(n)
    k = 2
    ev = np.concatenate([rng.uniform(0.5, 3.0, n - k), [30.0, 60.0]])
    W = _spectrum(n, ev, n + 1)
    p = n // 2
    d = si.mc_instance(p, n - p, 1, 4 * n, n)
    r = si.random_vec(d.m, 2)
    with SDPProblem.from_data(d, params=default_params(k=k)) as prob:
        prob.set_W(torch.from_numpy(W).cuda())
        prob.precond_build()
        tau, kk = prob.precond_info()
        z = prob.precond_apply(torch.from_numpy(r).cuda()).cpu().numpy()
    lo = ev.min()
    assert kk == k and abs(tau - lo) <= 4 * n * EPS * 60.0
    Q = []                                  # the top eigenvectors: unit vectors through the same reflections
    for t in (n - 2, n - 1):
        x = np.zeros(n)
        x[t] = 1.0
        g = np.random.default_rng(n + 1)
        for _ in range(3):
            h = g.standard_normal(n)
            h /= np.linalg.norm(h)
            x -= 2.0 * h * (h @ x)
        Q.append(x * np.sqrt(ev[t] - lo))
    U = np.stack(Q, 1)
    i, j = np.asarray(d.Ai), np.asarray(d.Aj)
    V = np.zeros((n, k))                    # V U
    np.add.at(V, i, 0.5 * z[:, None] * U[j])
    np.add.at(V, j, 0.5 * z[:, None] * U[i])
    Hz = lo * lo * 0.5 * z + 2.0 * lo * 0.5 * ((V[i] * U[j]).sum(1) + (V[j] * U[i]).sum(1))
    assert np.linalg.norm(Hz - r) <= 4 * n * EPS * (1 + 2 * 60.0 / lo) * np.linalg.norm(r)


@pytest.mark.parametrize("n", [1025, 2047])
def test_nt_scaling_above_order_1024(n):
    """All eigenvectors, back-transformed: W S W = X to 50 n eps kappa(X) kappa(S), kappa <= 4 each."""
    from paper_1703_10973_gb300 import SDPProblem
    rng = np.random.default_rng(n)
    X, S = _spectrum(n, rng.uniform(0.5, 2.0, n), 1), _spectrum(n, rng.uniform(0.5, 2.0, n), 2)
    with SDPProblem.from_data(si.unit_diag_instance(n)) as prob:
        prob.set_state(X, np.zeros(n), S, 0)
        info = prob.ipm_step()
        W = prob.get_W().cpu().numpy()
    assert info["nt_fallback"] == 0
    assert np.linalg.norm(W @ S @ W - X) <= 50 * n * EPS * 16.0 * np.linalg.norm(X)


@pytest.mark.parametrize("n", [63, 64, 255, 256, 257, 519, 1025])
def test_step_that_the_boundary_cuts(n):
    """X twenty times too large: the step to X_ii = 1 leaves the cone.  alpha = 0.9 / -(theta - bound)
    with bound <= 1e-3 |theta| and theta - bound <= lambda_min(L^-1 dX L^-T) up to rounding: between
    0.998 of 0.9 of the largest step and that, on both sides of the orders at which Lanczos changes."""
    from paper_1703_10973_gb300 import SDPProblem
    rng = np.random.default_rng(n)
    U, V = (rng.standard_normal((n, 8)) / np.sqrt(n) for _ in range(2))
    X, S = 20.0 * (0.7 * np.eye(n) + U @ U.T), 0.9 * np.eye(n) + V @ V.T
    with SDPProblem.from_data(si.unit_diag_instance(n)) as prob:
        prob.set_state(X, np.zeros(n), S, 0)
        a = prob.ipm_step()["alpha_p"]
        X1, _, _ = prob.get_solution()
    assert a < 1.0
    L = np.linalg.cholesky(X)
    D = np.linalg.solve(L, np.linalg.solve(L, (X1 - X) / a).T)
    amax = -1.0 / np.linalg.eigvalsh((D + D.T) / 2)[0]
    assert 0.9 * 0.998 * amax * (1 - 1e-7) <= a <= 0.9 * amax * (1 + 1e-7)
