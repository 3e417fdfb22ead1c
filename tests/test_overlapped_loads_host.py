"""Kernels launched over their predecessor's end read what that one writes by ordinary loads:
the read-only path (__ldg, or a load from a const __restrict__ parameter, which the compiler
may turn into one) is for data that nothing writes while the kernel lives.  A
reading of the sources, without a GPU."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1809_02390_gb300", "csrc")
# Parameters of batch kernels that are written once, before the first step.
FIXED = {"tiles", "coef", "maps"}


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def _kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__\b", text):
        head = re.compile(r"\b(k_\w+)\s*\(").search(text, m.end())
        depth, i = 1, head.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params, j = text[head.end():i - 1], text.index("{", i)
        depth, k = 1, j + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield head.group(1), params, text[j:k]


def test_no_read_only_loads_of_populations():
    overlapped = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = _code(path)
        for name, params, body in _kernels(text):
            if "follow_predecessor" in body:
                overlapped += 1
                assert "__ldg" not in body, name
                read_only = re.findall(r"const\s+[\w:<>]+\s*\*\s*__restrict__\s+(\w+)", params)
                assert set(read_only) <= FIXED, (name, read_only)
            text = text.replace(body, "")
        # Device functions: any kernel may call them.
        assert "__ldg" not in text, path
    assert overlapped >= 6
