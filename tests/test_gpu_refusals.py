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


def test_sampling_needs_an_output(qsim):
    """A NULL output is an invalid argument, whatever the number of shots."""
    import ctypes
    L, st = qsim.lib(), qsim.State(5, qsim.C64)
    st.set_basis(3)
    z = (ctypes.c_double * 5)()
    u = (ctypes.c_double * 1)(0.5)
    for shots in (0, 1):
        assert L.qsim_sample(st.h, 1, shots, None) == 1          # QSIM_EINVAL
        assert L.qsim_sample_uniforms(st.h, u, shots, None) == 1
        assert L.qsim_expect_z_and_sample(st.h, z, z, 1, shots, None) == 1
    out = (ctypes.c_uint64 * 1)()
    assert L.qsim_sample(st.h, 1, 0, out) == 0
    assert L.qsim_expect_z_and_sample(st.h, z, z, 1, 1, out) == 0 and out[0] == 3
