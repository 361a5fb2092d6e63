"""The Hessian product at the orders where its SpMM changes rows per CTA, warps and slices
(32 rows each), in every precision, against the oracle.  Tolerances as for the same products
elsewhere in the tests: 1e-12 (FP64), 2e-5 (FP32 W), 2e-2 (BF16 W), relative 2-norm."""
import numpy as np
import pytest

import sdp_inputs as si
from oracle import sdp_oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 2e-5, "bf16": 2e-2}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10973_gb300 import _build, load
    _build.build()
    load()


def _check(d, prec):
    from paper_1703_10973_gb300 import SDPProblem
    W = si.random_spd(d.n, 3, cond=100.0)
    v = si.random_vec(d.m, 4)
    with SDPProblem.from_data(d) as prob:
        prob.set_W(torch.from_numpy(W).cuda())
        hv = prob.hessian_matvec(torch.from_numpy(v).cuda(), prec=prec).cpu().numpy()
    ref = o.hessian_matvec(o.Problem.from_data(d), W, v)
    assert np.linalg.norm(hv - ref) <= TOL[prec] * np.linalg.norm(ref)


@pytest.mark.parametrize("prec", list(TOL))
@pytest.mark.parametrize("n", [2, 31, 32, 33, 97, 128, 129, 305, 513, 609])
def test_matvec_at_edge_orders(n, prec):
    p = max(1, n // 3)
    _check(si.mc_instance(p, n - p, 1, max(1, p * (n - p) // 3), n), prec)


@pytest.mark.parametrize("prec", list(TOL))
def test_matvec_with_rows_of_very_different_length(prec):
    """One dense row (length n), many of length one: slices much wider than most of their rows."""
    _check(si.mc_instance(1, 199, 1, 199, 3), prec)
