"""Source check: a kernel that may overlap its predecessor reads what that one wrote
by plain loads after its wait, never by loads that promise unchanging data."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_04178_gb300", "csrc")


def kernels():
    """(name, parameters, body) of every kernel that calls grid_dependency_wait."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__ void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(([^{;]*?)\)\s*\{",
                             text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            body = text[m.end():end]
            if "grid_dependency_wait()" in body:
                yield m.group(1), m.group(2), body


def test_the_overlapping_kernels_are_found():
    assert {"gemm_kernel", "prep_kernel", "amax_kernel", "model_grad_finish_kernel"} <= {k[0] for k in kernels()}


@pytest.mark.parametrize("name,params,body", list(kernels()), ids=[k[0] for k in kernels()])
def test_no_read_only_loads_after_the_wait(name, params, body):
    after = body.split("grid_dependency_wait()", 1)[1]
    for load in ("__ldg(", "ld.global.nc", "__ldcs(", "__ldlu("):
        assert load not in after, load
    for p in params.split(","):
        if "const" in p and "__restrict__" in p:
            pointer = re.search(r"(\w+)\s*$", p.strip()).group(1)
            assert not re.search(r"\b%s\b" % pointer, after), pointer
