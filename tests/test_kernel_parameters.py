"""What a kernel that may start before its predecessor has ended says about its inputs."""
import glob
import os
import re

from conftest import ROOT


def _kernels():
    """(file, name, parameter list) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2603_11243_b200", "csrc", "*.cu*"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[end], 0)
                end += 1
            yield os.path.basename(path), m.group(1), text[m.end():end - 1]


def test_no_input_is_declared_unwritten_while_the_kernel_lives():
    """const T *__restrict__ allows a load in front of griddepcontrol.wait, when the kernel before may
    still be writing what is read; every kernel here is launched that way."""
    found = list(_kernels())
    assert len(found) >= 14
    wrong = [(f, k, p.strip()) for f, k, params in found for p in params.split(",")
             if "__restrict__" in p and re.search(r"\bconst\b", p)]
    assert not wrong, wrong
