"""Rules of the CUDA sources that no run shows for certain."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_20334_b200", "csrc")


def kernels():
    """(file, name, parameter list, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            params, start = text[m.end():i - 1], text.index("{", i)
            depth, j = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[j], 0)
                j += 1
            yield os.path.basename(path), m.group(1), params, text[start:j]


def test_kernels_that_start_early_take_no_read_only_pointers():
    # such a kernel runs before its predecessor's writes are complete, and a const __restrict__ parameter
    # lets the compiler read through the path for data that does not change while the kernel runs
    found = 0
    for path, name, params, body in kernels():
        if "wait_for_predecessor()" in body:
            found += 1
            assert not re.search(r"const\s+[^,]*\*\s*__restrict__", params), (path, name)
    assert found >= 6
