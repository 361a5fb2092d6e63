"""The FP64 Hessian product over row lengths of V around its batches of eight entries, on both sides of
the orders and lengths at which the kernel of T = W V changes (192 and 304 rows; eight entries a row),
with rows that hold nothing.  1e-12 relative 2-norm, as for the product elsewhere in the tests."""
import numpy as np
import pytest

import sdp_inputs as si
from oracle import sdp_oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10973_gb300 import _build, load
    _build.build()
    load()


def _instance(n, length, empty):
    """Completion with `length` samples in each row, the columns in turn; the last `empty` rows have none."""
    p = n // 2
    q = n - p
    i = np.repeat(np.arange(p - empty), length)
    j = p + (np.tile(np.arange(length), p - empty) + i) % q
    order = np.lexsort((j, i))
    d = si.mc_instance(p, q, 1, len(i), 1)
    d.Ai[:], d.Aj[:] = i[order], j[order]
    return d


@pytest.mark.parametrize("empty", [0, 5])
@pytest.mark.parametrize("length", [1, 7, 8, 9, 15, 16, 17, 25])
@pytest.mark.parametrize("n", [64, 191, 192, 193, 304, 305, 513])
def test_row_lengths(n, length, empty):
    from paper_1703_10973_gb300 import SDPProblem
    d = _instance(n, length, empty)
    W, v = si.random_spd(n, 3, cond=100.0), si.random_vec(d.m, 4)
    with SDPProblem.from_data(d) as prob:
        prob.set_W(torch.from_numpy(W).cuda())
        hv = prob.hessian_matvec(torch.from_numpy(v).cuda()).cpu().numpy()
    ref = o.hessian_matvec(o.Problem.from_data(d), W, v)
    assert np.linalg.norm(hv - ref) <= 1e-12 * np.linalg.norm(ref)
