"""Properties of the CUDA sources that no run shows reliably (CPU)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_32831_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"/\*.*?\*/", " ", f.read(), flags=re.S)
    return re.sub(r"//[^\n]*", " ", text)


@pytest.mark.parametrize("name", sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh"))))
def test_dependent_launches_read_no_read_only_loads(name):
    """A kernel that waits for the launch before it (griddep_wait) is resident
    while that launch writes its inputs. Read-only (non-coherent) loads need
    data that is constant over the kernel's lifetime, and the wait does not
    order them: sources with such kernels use neither the intrinsic nor the
    instruction, and no restrict-qualified pointer a compiler may turn into it."""
    code = _code(name)
    if "griddep_wait();" not in code:
        return
    assert not re.findall(r"__ldg\s*\(|\.nc\b|__restrict__", code)
