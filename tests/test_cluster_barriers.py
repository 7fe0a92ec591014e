"""Every cluster barrier of the device code is of the aligned form, which all threads of a warp
must execute together: behind code of one lane or thread the warp has to be re-converged
(__syncwarp or __syncthreads) right before it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_03313_gb300", "csrc")


def test_aligned_cluster_barriers_follow_a_convergence():
    found = 0
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name), encoding="utf-8") as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"asm volatile\(\s*\"barrier\.cluster\.", text):
            found += 1
            before = text[:m.start()].rstrip()
            assert before.endswith(("__syncwarp();", "__syncthreads();")), (name, before[-120:])
    assert found > 0
