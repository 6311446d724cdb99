"""Calls that are refused: one-shot runs under stream capture, sampling without a place for the samples."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qsim(gpu_lib):
    from paper_2511_14664_gb300 import qsim as q
    return q


@pytest.mark.parametrize("n,kw", [(12, dict(mode=1)), (12, dict(mode=0)), (18, dict(mode=1)), (18, dict(mode=0))])
def test_one_shot_run_is_refused_under_capture(qsim, n, kw):
    """A run plans, waits and frees its plan: it reports an error under capture, leaves the capture as it was, and the
    handle works afterwards."""
    import torch
    c = W.brickwork(n, 3, seed=2)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        st = qsim.State(n, qsim.C64, stream=side)
        st.set_basis(0)
    side.synchronize()
    g = torch.cuda.CUDAGraph()
    x = torch.zeros(4, device="cuda")
    with torch.cuda.graph(g, stream=side):
        x += 1
        with pytest.raises(qsim.QsimError):
            st.run(c, **kw)
    g.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [1.0] * 4
    st.set_basis(0)
    st.run(c, **kw)
    assert float(np.max(np.abs(st.get_state() - oracle.run(c)))) <= 1e-5
