"""Inverse iteration with eight vectors per CTA (more than 592 vectors): chains of different
length in one warp, and solutions that pass 2^400, where four lanes rescale a vector together.

S is block diagonal with tridiagonal blocks and X = I, so the tridiagonal form is S itself and
falls apart into these blocks; W = S^(-1/2) by blocks.  Each block is conditioned below 16, so
W S W = X holds to 50 n eps 16 (as for the scaling of other well conditioned iterates)."""
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


def _blocks(sizes, scales, seed):
    rng = np.random.default_rng(seed)
    n = sum(sizes)
    S, at = np.zeros((n, n)), 0
    for b, s in zip(sizes, scales):
        d, e = rng.uniform(1.0, 2.0, b), rng.uniform(0.1, 0.3, b - 1)
        S[at:at + b, at:at + b] = s * (np.diag(d) + np.diag(e, 1) + np.diag(e, -1))
        at += b
    return S


def _scaling(S):
    from paper_1703_10973_gb300 import SDPError, SDPProblem
    n = len(S)
    with SDPProblem.from_data(si.unit_diag_instance(n)) as prob:
        prob.set_state(np.eye(n), np.zeros(n), S, 0)
        try:
            prob.ipm_step()   # W comes first; the Newton system of an iterate of such scales may be refused
        except SDPError:
            pass
        return prob.get_W().cpu().numpy()


@pytest.mark.parametrize("small", [1.0, 1e-106])
@pytest.mark.parametrize("order", [1, -1])
def test_chains_of_different_length(small, order):
    """Blocks of order 40 and 2 (and 1); with the factor 1e-106 a solution on a small block grows to
    1e121 and more, past 2^400, beside chains that do not."""
    sizes = ([40] * 14 + [2] * 23 + [1] * 3)[::order]
    S = _blocks(sizes, [small if b == 2 else 1.0 for b in sizes], 5)
    W = _scaling(S)
    n = len(S)
    assert n > 592
    assert np.linalg.norm(W @ S @ W - np.eye(n)) <= 50 * n * EPS * 16.0 * np.sqrt(n)
