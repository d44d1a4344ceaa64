"""Kernels that stop at entry on a recorded error, by their source.

The render's binning kernels return at once when the status word already holds an
error.  Where a kernel can also write that word, another block of the same launch may
write it while this block starts: threads that read it one by one can then disagree,
some warps leave, and the others go on with shared words that the absent warps never
wrote (digit and run counts that become shared and global addresses).  Such a kernel
has to decide as a block.  A race of this kind is shown from the source, never by
running it.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2505_18992_gb300", "csrc")
ENTRY = re.compile(r"^ *if \((.*\*(?:ws\.)?status != 0u.*)\) return;", re.M)


def _kernels(text):
    """(name, source) of every kernel definition, up to the closing brace in column 0."""
    for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\([^;{]*\)\s*\{", text):
        yield m.group(1), text[m.start():text.index("\n}\n", m.end())]


def _split_decisions(text):
    return [name for name, src in _kernels(text)
            if "set_status(" in src and any("__syncthreads_or(" not in e for e in ENTRY.findall(src))]


def test_the_check_sees_a_split_decision():
    kernel = ("__global__ void k(uint32_t *status) {\n    if (%s) return;\n    __syncthreads();\n"
              "    set_status(status, 1);\n}\n")
    assert _split_decisions(kernel % "*status != 0u") == ["k"]
    assert _split_decisions(kernel % "lb.stop && *status != 0u") == ["k"]
    assert _split_decisions(kernel % "__syncthreads_or(*status != 0u)") == []


@pytest.mark.parametrize("unit", ["render_bin.cu", "prims.cuh"])
def test_kernels_that_write_the_status_word_enter_as_a_block(unit):
    with open(os.path.join(CSRC, unit)) as f:
        text = f.read()
    assert sum("set_status(" in src for _, src in _kernels(text)) > 0
    assert _split_decisions(text) == []
