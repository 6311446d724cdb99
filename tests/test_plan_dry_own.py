"""A dry run plans the passes that a plan in the state's own precision has: from 17 qubits on its blocks have at most 5
qubits, whatever width up to 6 is asked for."""
import pytest

import workloads as W


@pytest.mark.parametrize("dtype,precision", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("n", [16, 17, 20])
def test_dry_run_of_width_six(dtype, precision, n):
    from paper_2511_14664_gb300 import qsim
    c = W.brickwork(n, 8, seed=1)
    def passes(k):
        return qsim.Plan(c, dtype, mode=1, max_fused=k, precision=precision, dry_run=True).passes()
    six = passes(6)
    assert max(q["k"] for q in six) == (6 if n < 17 else 5)
    if n >= 17:
        assert six == passes(5)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n", [14, 18])
def test_dry_run_lists_the_plans_passes(gpu_lib, dtype, n):
    from paper_2511_14664_gb300 import qsim
    c = W.brickwork(n, 8, seed=1)
    for k in (5, 6):
        dry = qsim.Plan(c, dtype, mode=1, max_fused=k, dry_run=True).passes()
        assert dry == qsim.Plan(c, dtype, mode=1, max_fused=k).passes()
