"""The chain's kernels may start while the kernel that writes their input still runs, so they
read it by plain loads: __ldg asks for data that does not change while the kernel runs.
Masks, and the fields of the stage calls, are in place before any kernel that reads them starts."""
import os
import re

import pytest

from paper_2508_07476_gb300 import build

STEADY = r"(reinterpret_cast<const (uint32_t|float4)\*>\()?(mask|evals|evec)\b"


@pytest.mark.parametrize("name", ["ct_k_eig.cu", "ct_k_grad2.cu", "ct_k_rho.cu", "ct_k_rhoxy.cu", "ct_k_rhotc.cu"])
def test_chain_inputs_are_read_by_plain_loads(name):
    with open(os.path.join(build.CSRC, name)) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    assert "after_previous(" in code
    assert [m for m in re.findall(r"__ldg\(([^;]*);", code) if not re.match(STEADY, m)] == []
    if name == "ct_k_rhotc.cu":  # element copies of the gradient
        assert not re.search(r"= gbase\[", code)
