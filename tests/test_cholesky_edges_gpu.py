"""Cholesky factors at orders around its 32-column panels (one panel, a full and a ragged one,
several), by the scaling matrix that an iteration forms from chol(X) and chol(S):
W = X^1/2 (X^1/2 S X^1/2)^-1/2 X^1/2.  With eigenvalues of X and S in [1, 4] the condition of every
factor is at most 4, of the product 16, so n eps 16 < 1e-11 bounds the error."""
import numpy as np
import pytest

import sdp_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sqrt(A, power=0.5):
    w, Q = np.linalg.eigh(A)
    return (Q * w ** power) @ Q.T


@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 63, 64, 65, 97, 130, 257])
def test_scaling_matrix(n):
    from paper_1703_10973_gb300 import SDPProblem, _build, load
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _build.build()
    load()
    p = max(1, n // 3)
    d = si.mc_instance(p, n - p, 1, max(1, p * (n - p) // 2), n)
    X, S = si.random_spd(n, 1, cond=4.0), si.random_spd(n, 2, cond=4.0)
    with SDPProblem.from_data(d) as prob:
        prob.set_state(X, np.zeros(d.m), S)
        prob.ipm_step()
        W = prob.get_W()
    W = W.cpu().numpy() if hasattr(W, "cpu") else np.asarray(W)
    R = _sqrt(X)
    M = R @ S @ R
    ref = R @ _sqrt((M + M.T) / 2, -0.5) @ R
    assert np.linalg.norm(W.reshape(n, n) - ref) <= 1e-11 * np.linalg.norm(ref)
