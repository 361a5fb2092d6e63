"""Build and apply of the Hhat preconditioner where its kernels change shape: split ranks 1 to 8
and above, independent sets of a few vertices and of more than a CTA's width, rows with more
neighbours than a pass of the Schur complement stages, general constraints.  Against the oracle's
dense matrix; tolerance 20 cond(Hhat) eps, as for the same solve elsewhere in the tests."""
import numpy as np
import pytest

import sdp_inputs as si
from oracle import sdp_oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = {
    "one_by_one": (lambda: si.mc_instance(1, 1, 1, 1, 1), (1,)),
    "star": (lambda: si.mc_instance(1, 140, 1, 140, 2), (1, 3)),
    "few": (lambda: si.mc_instance(3, 66, 1, 150, 3), (1, 4, 8)),
    "square": (lambda: si.mc_instance(33, 31, 1, 700, 4), (2, 5, 7, 9)),
    "many_neighbours": (lambda: si.mc_instance(150, 9, 1, 1200, 5), (1, 6, 8)),
    "long_rows": (lambda: si.mc_instance(300, 320, 1, 1500, 6), (8,)),
    "general": (lambda: si.random_general(23, 40, 3, 2), (1, 3, 8)),
    "diag": (lambda: si.diag_constraint_instance(17, 1), (1, 2)),
}


@pytest.mark.parametrize("case,k", [(c, k) for c in CASES for k in CASES[c][1]])
def test_hat_against_the_dense_matrix(case, k):
    from paper_1703_10973_gb300 import SDPProblem, _build, default_params, load
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _build.build()
    load()
    d = CASES[case][0]()
    k = min(k, d.n - 1)
    rng = np.random.default_rng(k)
    Q, _ = np.linalg.qr(rng.standard_normal((d.n, d.n)))
    W = (Q * np.concatenate([rng.uniform(1.0, 3.0, d.n - k), rng.uniform(1.0, 2.0, k) / 1e-2])) @ Q.T
    r = si.random_vec(d.m, 2)
    P = o.Problem.from_data(d)
    with SDPProblem.from_data(d, params=default_params(precond=2, k=k)) as prob:
        prob.set_W(torch.from_numpy(W).cuda())
        prob.precond_build()
        z = prob.precond_apply(torch.from_numpy(r).cuda()).cpu().numpy()
    Hh = o.precond_dense(P, o.precond_hat_build(P, W, k))
    x = np.linalg.solve(Hh, r)
    tol = max(1e-12, 20.0 * np.linalg.cond(Hh) * np.finfo(float).eps)
    assert np.linalg.norm(z - x) <= tol * np.linalg.norm(x)
