"""A kernel whose launch overlaps the grid before it (it begins with chain_wait) must not read through the read-only
path what that grid may still be writing: no __ldg, no const __restrict__ parameter, no read-only load policy."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_08643_gb300", "csrc")
KERNEL = re.compile(r"__global__ void (?:__launch_bounds__\([^)]*\) )?(\w+)\(([^{]*)\)\s*\{\s*chain_wait\(\);(.*?)\n\}\n", re.S)


def _chained():
    for name in ("lbm_kernels.cu", "lbm_kernels_pair.cu"):
        with open(os.path.join(CSRC, name)) as fh:
            for kernel, params, body in KERNEL.findall(fh.read()):
                yield pytest.param(params, body, id=kernel)


def test_every_chained_kernel_is_looked_at():
    assert len(list(_chained())) == 6


@pytest.mark.parametrize("params, body", list(_chained()))
def test_no_read_only_loads(params, body):
    inputs = [p for p in params.split(",") if "const" in p and "*" in p]
    assert inputs and not any("__restrict__" in p for p in inputs)
    assert "__ldg" not in body and "PairIO" not in body and "pull_q<Q, true" not in body
    assert "PlainLoad" in body or "pull_q<Q, false" in body
