"""Circuits of 19 qubits and more with no fusion width given: clusters or plans of their own, whichever is estimated faster,
take no longer than 1.25 times as the clusters alone (which a given fusion width asks for), medians of the same run."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,make", [
    (0, lambda: [W.rcs(19, i, gates_per_qubit=10) for i in range(40)]),
    (0, lambda: [W.random_pairs(19, 6, i) for i in range(40)]),
    (0, lambda: [W.brickwork(20, 6, i) for i in range(12)]),
    (0, lambda: [W.tfim_chain(19 + i % 3, 8, 0.4 + 0.05 * i, 0.8) for i in range(9)]),
    (4, lambda: [W.rcs(19, i, gates_per_qubit=10) for i in range(30)] + [W.rcs(22, 70 + i, gates_per_qubit=10) for i in range(4)]),
    (4, lambda: [W.random_pairs(19, 6, i) for i in range(30)] + [W.random_pairs(22, 6, 70 + i) for i in range(4)])])
def test_no_slower_than_clusters(gpu_lib, precision, make):
    import torch
    from paper_2511_14664_gb300 import qsim
    cs = make()

    def median(**kw):
        b = qsim.Batch(cs, precision=precision, **kw)
        times = []
        for _ in range(11):
            s, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            s.record()
            b.execute()
            e.record()
            torch.cuda.synchronize()
            times.append(s.elapsed_time(e))
        b.close()
        return sorted(times[2:])[4]

    assert median(max_fused=0) <= 1.25 * median(max_fused=4)
