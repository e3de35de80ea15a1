"""A function's execution space must not depend on __CUDA_ARCH__: nvcc compiles a kernel's source once for the host
and once for the device, and both have to see the same declarations."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_09733_gb300", "csrc")


def test_no_declaration_is_chosen_by_the_compilation_pass():
    for name in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, name)).read()
        for part in re.findall(r"#if[^\n]*__CUDA_ARCH__.*?#endif", src, re.S):
            assert "__device__" not in part and "inline" not in part, name
