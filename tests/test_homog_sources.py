"""The rate equations divide by CUDA's own rounded operations: no FP32 reciprocal seeds, and no
FP32 arithmetic in the error estimate and the step-size control."""
import os
import re

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_03313_gb300", "csrc",
                      "homog.cu")


def _code():
    with open(SOURCE, encoding="utf-8") as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_reciprocals_are_rounded_ones():
    code = _code()
    assert "__frcp_rn" not in code and "hx_recip" not in code
    assert "__drcp_rn" in code
