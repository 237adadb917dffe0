"""Kernels that may be set up while the kernel before them still runs (they begin with griddep_wait()): what a call is given or an earlier
kernel writes is not read by the non-coherent path, which is for memory that nothing writes while the grid is there.  Only the model's own
arrays are.  Read from the sources: what a compiler makes of such a load may change without a line of them changing."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_24174_b200", "csrc")
CONSTANT = {"embed", "gain"}                                                          # parameters
LDG = r"w0|w1|a\.embed|a\.gain|ph\.gain|gain"                                         # and what __ldg may be given


def sources_with_waits():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = "\n".join(line.split("//", 1)[0] for line in open(path))
        if "griddep_wait()" in text:
            yield path, text


def kernels(text):
    """(name, parameters, body up to the next kernel) of every kernel that waits for the one before it."""
    starts = list(re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\s*\(([^{;]*)\)\s*\{", text))
    for m, after in zip(starts, starts[1:] + [None]):
        body = text[m.end():after.start() if after else len(text)]
        if "griddep_wait()" in body:
            yield m.group(1), m.group(2), body


def test_the_kernels_are_found():
    names = {name for _, text in sources_with_waits() for name, _, _ in kernels(text)}
    assert {"draft_kernel", "rows_embed_kernel", "accept_kernel", "forward_f32_kernel", "attn_mma_kernel", "gemm_wide_kernel"} <= names


@pytest.mark.parametrize("path", [p for p, _ in sources_with_waits()], ids=os.path.basename)
def test_only_constant_arrays_are_read_by_the_non_coherent_path(path):
    text = dict(sources_with_waits())[path]
    for name, parameters, body in kernels(text):
        read_only = set(re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", parameters))
        assert read_only <= CONSTANT, (name, read_only - CONSTANT)
        for given in re.findall(r"__ldg\((?:reinterpret_cast<[^>]*>\()?\s*([\w.]+)", body):
            assert re.fullmatch(LDG, given), (name, given)
