"""Compile-time knobs of the CUDA library that a build cannot honour are refused by the
compiler, with the reason, instead of giving wrong results or failing calls later."""
import os
import subprocess

import pytest

from paper_2505_18992_gb300 import build as B


def _compile(unit, flags, out):
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc here")
    return subprocess.run([nvcc, *B.ARCH, *B.NVCC_FLAGS, *flags, "-c", os.path.join(B.CSRC, unit), "-o", str(out)],
                          capture_output=True, text=True)


@pytest.mark.parametrize("unit,flag,reason", [
    ("render_comp.cu", "-DVPGS_FWD_BATCH=4", "16-bit offsets"),
    ("render_comp.cu", "-DVPGS_BWD_BATCH=4", "16-bit offsets"),
    ("render_comp.cu", "-DVPGS_GEO_BATCH=4", "16-bit offsets"),
    ("api.cu", "-DVPGS_PIX=1", "two rows per thread"),
    ("render_comp.cu", "-DVPGS_PIX=4", "two rows per thread"),
    ("render_bin.cu", "-DVPGS_DEPTH_SORT_ITEMS=5", "keys per thread"),
    ("render_bin.cu", "-DVPGS_TILE_SORT_ITEMS=64", "keys per thread"),
])
def test_refused_at_compile_time(unit, flag, reason, tmp_path):
    res = _compile(unit, [flag], tmp_path / "unit.o")
    assert res.returncode != 0 and reason in res.stderr, res.stderr
