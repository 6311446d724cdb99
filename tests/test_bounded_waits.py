"""Kernels whose roles leave on an expired wait hold no wait without a limit among those roles.

A warp that gives up goes to the end of the kernel; a named barrier (bar.sync) that counts it would then keep its
neighbours for ever. (Read from the source: such a wait is not provoked on a GPU.)"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_14664_gb300", "csrc")


@pytest.mark.parametrize("name", ["k_tcx.cu", "k_tc_pair.cu", "k_tc.cu", "k_tc7.cu"])
def test_no_named_barrier_beside_bounded_waits(name):
    text = open(os.path.join(CSRC, name)).read()
    assert "mbar_wait_bounded" in text
    code = re.sub(r"//[^\n]*", "", text)
    assert not re.search(r"\b(bar|barrier)\.(cta\.)?(sync|red)\b|__barrier_sync|named_barrier", code)
