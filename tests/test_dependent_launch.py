"""Kernels that wait on the kernel before them (griddepcontrol.wait) are resident
while it still writes its results.  A `const T* __restrict__` parameter
promises data that nothing writes during the kernel's life, and allows
non-coherent loads, which the wait does not order: such a kernel takes plain
pointers.  Read from the sources, since a stale load cannot be provoked."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_10516_gb300", "csrc")
KERNEL = re.compile(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(")


def _span(text, start, opener, closer):
    """The text between the bracket at `start` and its match."""
    depth = 0
    for i in range(start, len(text)):
        depth += (text[i] == opener) - (text[i] == closer)
        if depth == 0:
            return text[start + 1:i], i
    raise AssertionError("unbalanced " + opener)


def _dependent_kernels():
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in KERNEL.finditer(text):
            params, end = _span(text, m.end() - 1, "(", ")")
            body, _ = _span(text, text.index("{", end), "{", "}")
            if "pdl_wait()" in body or "griddepcontrol.wait" in body:
                out.append((os.path.basename(path), m.group(1), params))
    return out


def test_dependent_kernels_are_found():
    names = {k for _, k, _ in _dependent_kernels()}
    assert {"cheb_step_kernel", "cheb_long_kernel", "reduce_partials_kernel", "mlp_tile_kernel", "mlp_reduce_kernel",
            "mlp_reduce_adam_kernel"} <= names


@pytest.mark.parametrize("path,name,params", _dependent_kernels(), ids=lambda x: x if "(" not in x and " " not in x else "")
def test_no_read_only_parameters(path, name, params):
    assert not re.search(r"const\s[^,]*\*\s*__restrict__", params), (path, name)
