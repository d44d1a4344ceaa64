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


LAYOUT = r'''
#include "%s/api.cu"
#include <stdio.h>
int main() {
    vpgs_render_opts o;
    memset(&o, 0, sizeof(o));
    o.tile_w = o.tile_h = 16;
    o.alpha_min = 0.01f; o.alpha_max = 0.99f; o.t_min = 1e-4f; o.dilation = 0.3f; o.near_z = 0.2f;
    const int sizes[][2] = {{97, 61}, {320, 240}, {800, 900}, {3840, 2160}};
    for (int V = 1; V <= 4; V += 3)
        for (auto &wh : sizes)
            for (int64_t N = 1; N <= 13000; N += N < 20 ? 1 : 61) {
                vpgs_camera cam = {wh[0], wh[1], 100.f, 100.f, 50.f, 50.f};
                RenderLayout L;
                if (!make_layout(N, V, &cam, &o, 64, L)) { printf("no layout\n"); return 0; }
                if (bin_form(L) == kGeneralBin) continue;
                // what a small call keeps in the depth sort's buffers: a word per pair each
                const size_t need = 4 * (size_t)L.VN;
                if (L.off_sort_look_t - L.off_sort_look < need || L.off_dval0 - L.off_dkey0 < need ||
                    L.off_dkey1 - L.off_dval0 < need || L.off_dval1 - L.off_dkey1 < need ||
                    L.off_ikey0 - L.off_dval1 < need) {
                    printf("too small: %%d views of %%lld at %%dx%%d\n", V, (long long)N, wh[0], wh[1]);
                    return 0;
                }
            }
    printf("fits\n");
    return 0;
}
'''


@pytest.mark.parametrize("flags", [[], ["-DVPGS_DEPTH_SORT_ITEMS=8"], ["-DVPGS_DEPTH_SORT_ITEMS=16"]])
def test_buffers_borrowed_by_small_calls_hold_them(flags, tmp_path):
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc here")
    src, exe = tmp_path / "layout.cu", tmp_path / "layout"
    src.write_text(LAYOUT % B.CSRC)
    # only the host's layout runs; the launches that api.cu calls stay unresolved
    res = subprocess.run([nvcc, *B.ARCH, *B.NVCC_FLAGS, *flags, str(src), "-o", str(exe), "-cudart", "static",
                          "-Xlinker", "--unresolved-symbols=ignore-all"], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.stdout == "fits\n", (out.stdout, out.stderr)
