"""Kernels that may start before the kernel in front of them has finished
(launch_after, after_wait in irs_common.cuh) must not declare what that kernel
writes `const __restrict__`: the qualifier promises data that nobody writes
while the kernel lives.  Read from the sources: no GPU needed."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_10871_gb300", "csrc")

# complete before the first kernel of a call: the caller's inputs and the plan's tables
COMPLETE = {"xy", "mass", "idx", "tw", "kspec_d", "kspec_f", "sheet_d", "sheet_f", "sheet_near"}


def _chained_kernels():
    text = "\n".join(open(f).read() for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))
    launched = set(re.findall(r"launch_after\(\s*(?:\w+ \? )?(k_\w+)", text))
    launched |= set(re.findall(r"auto\* kern = \w+ \? (k_\w+)", text))
    heads = dict(re.findall(r"__global__ void[^;{]*?\b(k_\w+)\(([^{]*?)\)\s*\{", text))
    return {k: heads[k] for k in launched}


def test_every_chained_kernel_is_found():
    assert len(_chained_kernels()) >= 12


@pytest.mark.parametrize("kernel", sorted(_chained_kernels()))
def test_inputs_written_in_the_chain_are_plain_pointers(kernel):
    read_only = set(re.findall(r"const \w+\* __restrict__ (\w+)", _chained_kernels()[kernel]))
    assert read_only <= COMPLETE, sorted(read_only - COMPLETE)
