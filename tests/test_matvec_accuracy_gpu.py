"""The FP64 Hessian product is a double-precision product entry by entry, whatever the scales of W and
v, and reads the W of its time.

Bound.  Hv_i is a sum of products W_pk V_kl W_lq; summed in double in any order, its error is at most
N u times the sum of their magnitudes (|A| |W| |V| |W|)_i, u = 2^-53, with N the roundings on the way
of a product: below n + (largest row of V) + (entries of A_i) + 8.  The reference is formed in long double."""
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


def _wide(d, W, v):
    """Hv and the sums of magnitudes, in long double."""
    i, j, k = (np.asarray(x) for x in (d.Ai, d.Aj, d.Ak))
    off, x = i != j, np.asarray(d.Av).astype(np.longdouble)
    out = []
    for mag in (False, True):
        f = np.abs if mag else (lambda a: a)
        Wl, val = f(W.astype(np.longdouble)), f(x * v[k])
        T = np.zeros((d.n, d.n), np.longdouble)   # (V W), a row per entry of V
        np.add.at(T, i, val[:, None] * Wl[j])
        np.add.at(T, j[off], val[off, None] * Wl[i[off]])
        dots = (Wl[i] * T[:, j].T).sum(1)         # (W V W)_ij
        hv = np.zeros(d.m, np.longdouble)
        np.add.at(hv, k, f(x) * np.where(off, 2, 1) * dots)
        out.append(hv)
    rows = np.bincount(np.concatenate([i, j[off]]), minlength=d.n).max()
    return out[0], out[1], d.n + rows + np.bincount(k).max() + 8


def _check(d, W, v):
    from paper_1703_10973_gb300 import SDPProblem
    with SDPProblem.from_data(d) as prob:
        prob.set_W(torch.from_numpy(np.ascontiguousarray(W)).cuda())
        hv = prob.hessian_matvec(torch.from_numpy(v).cuda()).cpu().numpy()
    ref, mag, N = _wide(d, W, v)
    assert np.all(np.abs(hv - ref) <= N * 2.0 ** -53 * mag)


def _drop(d, index):
    """The instance without the samples of one index."""
    keep = (np.asarray(d.Ai) != index) & (np.asarray(d.Aj) != index)
    m = int(keep.sum())
    return si.SDPData(n=d.n, m=m, Ci=d.Ci, Cj=d.Cj, Cv=d.Cv, Ak=np.arange(m, dtype=np.int32),
                      Ai=d.Ai[keep], Aj=d.Aj[keep], Av=d.Av[keep], b=d.b[keep], k=d.k)


@pytest.mark.parametrize("sampled", [True, False])
@pytest.mark.parametrize("big", [1e3, 1e6, 1e8])
def test_one_dominating_index(big, sampled):
    d = si.mc_instance(90, 111, 1, 1200, 1)
    if not sampled:
        d = _drop(d, 30)
    D = np.ones(d.n)
    D[30] = big
    _check(d, si.random_spd(d.n, 3, cond=100.0) * D[:, None] * D[None, :], si.random_vec(d.m, 4))


@pytest.mark.parametrize("s", [2, 4, 6])
def test_two_classes_of_different_scale(s):
    p, q = 80, 150
    d = si.mc_instance(p, q, 1, 4000, 2)
    D = np.concatenate([np.full(p, 10.0 ** s), np.full(q, 10.0 ** -s)])
    _check(d, si.random_spd(d.n, 3, cond=100.0) * D[:, None] * D[None, :], si.random_vec(d.m, 4))


@pytest.mark.parametrize("make", [lambda: si.mc_instance(100, 110, 1, 3000, 3), lambda: si.random_general(230, 60, 5, 2)],
                         ids=["completion", "general"])
@pytest.mark.parametrize("W", ["identity", "diagonal", "dense"])
def test_v_of_very_different_size(make, W):
    """Entries of v over twenty decades: an entry of V far below its neighbours in the row counts."""
    d = make()
    rng = np.random.default_rng(5)
    M = {"identity": np.eye(d.n), "diagonal": np.diag(10.0 ** rng.uniform(-6, 6, d.n)),
         "dense": si.random_spd(d.n, 3, cond=100.0)}[W]
    _check(d, M, si.random_vec(d.m, 4) * 10.0 ** rng.uniform(-10, 10, d.m))


@pytest.mark.parametrize("n", [300, 1217])
def test_evenly_scaled(n):
    p = n // 3
    d = si.mc_instance(p, n - p, 1, 6 * n, n)
    _check(d, si.random_spd(n, 3, cond=100.0), si.random_vec(d.m, 4))


def test_replayed_set_W_is_seen():
    """sdp_set_W is a copy on the handle's stream and may be captured: a replay changes the scaling
    matrix of the products and solves that follow it."""
    from paper_1703_10973_gb300 import SDPProblem, default_params
    d = si.mc_instance(100, 130, 1, 3000, 8)
    P, v = o.Problem.from_data(d), si.random_vec(d.m, 4)
    rng = np.random.default_rng(1)
    U = 3.0 * np.linalg.qr(rng.standard_normal((d.n, 1)))[0]
    Ws = [si.random_spd(d.n, s, cond=3.0) + s * U @ U.T for s in (1, 2, 3)]
    st = torch.cuda.Stream()
    with torch.cuda.stream(st), SDPProblem.from_data(d, params=default_params(k=1), stream=st.cuda_stream) as prob:
        buf, vd = torch.from_numpy(Ws[0]).cuda(), torch.from_numpy(v).cuda()
        prob.set_W(buf)
        prob.precond_build()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            prob.set_W(buf)
        for W in Ws:
            buf.copy_(torch.from_numpy(W))
            g.replay()
            hv = prob.hessian_matvec(vd).cpu().numpy()
            ref = o.hessian_matvec(P, W, v)
            assert np.linalg.norm(hv - ref) <= 1e-12 * np.linalg.norm(ref)
            y, _, rel, _ = prob.pcg_solve(vd, rtol=1e-9, maxit=2000)
            res = v - o.hessian_matvec(P, W, y.cpu().numpy())
            assert rel <= 1e-9 and np.linalg.norm(res) <= 1.1e-9 * np.linalg.norm(v)
