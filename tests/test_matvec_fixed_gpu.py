"""The fixed-point form of the FP64 Hessian product (orders above 192): edge orders, shared slots,
values of very different size, infinities and NaN, captured calls, PCG.  Tolerances as for the
product and the solve elsewhere in the tests: 1e-12 relative 2-norm, the requested residual."""
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


def _product(d, W, v):
    from paper_1703_10973_gb300 import SDPProblem
    with SDPProblem.from_data(d) as prob:
        prob.set_W(torch.from_numpy(W).cuda())
        return prob.hessian_matvec(torch.from_numpy(v).cuda()).cpu().numpy()


def _mc(n, seed, m=None):
    p = n // 3
    return si.mc_instance(p, n - p, 1, m or p * (n - p) // 3, seed)


@pytest.mark.parametrize("n", [193, 194, 223, 224, 225, 289, 303, 304, 305, 513, 609, 1217])
def test_edge_orders(n):
    d = _mc(n, n)
    W, v = si.random_spd(n, 3, cond=100.0), si.random_vec(d.m, 4)
    ref = o.hessian_matvec(o.Problem.from_data(d), W, v)
    assert np.linalg.norm(_product(d, W, v) - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("make", [lambda: si.random_general(230, 60, 5, 2), lambda: si.unit_diag_instance(201),
                                  lambda: si.mc_instance(1, 240, 1, 240, 3)], ids=["general", "unit_diag", "star"])
def test_patterns(make):
    d = make()
    W, v = si.random_spd(d.n, 3, cond=100.0), si.random_vec(d.m, 4)
    ref = o.hessian_matvec(o.Problem.from_data(d), W, v)
    assert np.linalg.norm(_product(d, W, v) - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("scale", [1e-300, 1e-160, 1.0, 1e140])
@pytest.mark.parametrize("spread", [0.0, 3.0])
def test_scaled_rows(scale, spread):
    """Rows of W and entries of v over many powers of ten; results down to subnormals and zero."""
    d = _mc(211, 5)
    rng = np.random.default_rng(6)
    D = 10.0 ** rng.uniform(-spread, spread, d.n)
    W = si.random_spd(d.n, 3, cond=100.0) * D[:, None] * D[None, :]
    v = si.random_vec(d.m, 4) * 10.0 ** rng.uniform(-spread, spread, d.m)
    s = np.sqrt(abs(scale)) if scale < 1e-200 else 1.0
    ref = o.hessian_matvec(o.Problem.from_data(d), W, v)
    got = _product(d, W * s, v * (scale if s == 1.0 else 1.0))
    assert np.linalg.norm(got / scale - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("where", ["W", "v"])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_infinities_and_nan(where, bad):
    """Entries that touch no infinity or NaN keep their values, the others are what FP64 sums give."""
    import scipy.sparse as sp
    d = _mc(199, 7, m=150)
    W, v = si.random_spd(d.n, 3, cond=100.0), si.random_vec(d.m, 4)
    if where == "W":
        W[5, 90] = W[90, 5] = bad
    else:
        v[17] = bad
    i, j, k = np.asarray(d.Ai), np.asarray(d.Aj), np.asarray(d.Ak)
    x = np.asarray(d.Av) * v[k]
    off = i != j
    V = sp.csr_matrix((np.concatenate([x, x[off]]), (np.concatenate([i, j[off]]), np.concatenate([j, i[off]]))),
                      shape=(d.n, d.n))
    with np.errstate(invalid="ignore"):
        T = (V.T @ W.T).T                      # stored entries only, as the kernels
        ref = np.zeros(d.m)
        for a in range(len(k)):
            s = (W[i[a]] * T[j[a]]).sum() if not off[a] else (W[i[a]] * T[j[a]]).sum() + (W[j[a]] * T[i[a]]).sum()
            ref[k[a]] += d.Av[a] * s
    got = _product(d, W, v)
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), fin)
    assert np.linalg.norm(got[fin] - ref[fin]) <= 1e-12 * max(np.linalg.norm(ref[fin]), 1e-300)


def test_captured_call_reads_the_W_of_its_replay():
    from paper_1703_10973_gb300 import SDPProblem
    d = _mc(205, 8)
    P, v = o.Problem.from_data(d), si.random_vec(d.m, 4)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st), SDPProblem.from_data(d, stream=st.cuda_stream) as prob:
        vd, out = torch.from_numpy(v).cuda(), torch.empty(d.m, dtype=torch.float64, device="cuda")
        prob.set_W(torch.from_numpy(si.random_spd(d.n, 1, cond=10.0)).cuda())
        prob.hessian_matvec(vd, out=out)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            prob.hessian_matvec(vd, out=out)
        W = si.random_spd(d.n, 2, cond=10.0)
        prob.set_W(torch.from_numpy(W).cuda())
        g.replay()
        st.synchronize()
        again = prob.hessian_matvec(vd).cpu().numpy()
        ref = o.hessian_matvec(P, W, v)
        assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
        assert np.linalg.norm(again - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_pcg(graph, prec):
    from paper_1703_10973_gb300 import SDPProblem, default_params
    d = _mc(230, 9, m=2000)
    P = o.Problem.from_data(d)
    rng = np.random.default_rng(1)
    U = rng.standard_normal((d.n, 2))
    r = si.random_vec(d.m, 2)
    with SDPProblem.from_data(d, params=default_params(precond=2, k=2, pcg_graph=graph, prec=prec)) as prob:
        for seed in (1, 2):   # the second W has to reach the limbs and the graph
            W = si.random_spd(d.n, seed, cond=3.0) + U @ U.T
            prob.set_W(torch.from_numpy(W).cuda())
            y, its, rel = prob.pcg_solve(torch.from_numpy(r).cuda(), rtol=1e-10, maxit=500, prec=prec)[:3]
            res = r - o.hessian_matvec(P, W, y.cpu().numpy())
            assert np.linalg.norm(res) <= 1.1e-10 * np.linalg.norm(r)
