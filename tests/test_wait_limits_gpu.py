"""params.wait_cycles bounds the waits of the whole-GPU Lanczos (step lengths from order 256 on): given
almost no time, the call reports SDP_ERR_TIMEOUT and the library stays usable."""
import numpy as np
import pytest

import sdp_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10973_gb300 import _build, load
    _build.build()
    load()


def test_step_length_wait_runs_out():
    from paper_1703_10973_gb300 import SDPError, SDPProblem, _lib, default_params
    d = si.mc_instance(150, 150, 1, 3000, 31)
    with SDPProblem.from_data(d, params=default_params(wait_cycles=1)) as p:
        with pytest.raises(SDPError) as e:
            p.ipm_step()
        assert e.value.status == _lib.SDP_ERR_TIMEOUT
        assert "timeout" in p.lib.sdp_last_error(p.h).decode()
    with SDPProblem.from_data(d) as p:
        info = p.ipm_step()
        assert info["pcg_relres_pred"] <= 1e-8 and np.isfinite(info["mu"])
