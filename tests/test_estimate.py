"""The admission estimate is an upper bound of what a problem holds on the device, and near it."""
import dataclasses

import numpy as np
import pytest

import sdp_inputs as si
from paper_1703_10973_gb300.serve import estimate_request_bytes

FIXED = 8 << 20   # the estimate's allowance


def test_malformed_requests_are_left_to_setup():
    d = si.mc_instance(20, 30, 1, 200, 1)
    for bad in (dict(Ak=np.where(np.arange(200) == 5, -3, d.Ak)), dict(Ak=d.Ak[:-1]), dict(Ak=d.Ak + 10 ** 6), dict(m=0)):
        assert estimate_request_bytes(dataclasses.replace(d, **bad)) > 0


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("make", [
    lambda: si.mc_instance(20, 20, 1, 200, 1), lambda: si.mc_instance(1, 240, 1, 240, 2),
    lambda: si.mc_instance(50, 400, 4, 10000, 3), lambda: si.mc_instance(400, 400, 4, 80000, 4),
    lambda: si.mc_instance(100, 900, 1, 2000, 5), lambda: si.random_general(200, 300, 20, 6),
    lambda: si.unit_diag_instance(300)],
    ids=["tiny", "star", "wide", "dense", "sparse", "general", "diagonal"])
def test_bounds_what_a_problem_holds(make, prec):
    """Twice the bytes at most, beside the fixed allowance."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10973_gb300 import SDPError, SDPProblem, _build, default_params, load
    _build.build()
    load()
    d = make()
    with SDPProblem.from_data(d, params=default_params(prec=prec)) as p:
        try:
            p.ipm_step()
        except SDPError:
            pass
        p.hessian_matvec(torch.ones(d.m, dtype=torch.float64, device="cuda"), prec=prec)
        held = p.device_bytes()
    assert held <= estimate_request_bytes(d) <= FIXED + 2 * held
