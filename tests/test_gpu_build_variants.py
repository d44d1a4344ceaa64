"""Builds of the library with other compile-time knobs, on the GPU against the default build.

Each variant is a copy of the package compiled with VPGS_NVCC_FLAGS and run in a
process of its own on the same inputs.  One scene is a single tile of 64 pixels, where
each sum has one order and so one result; the others are large enough for the general
binning (scans, both radix sorts, emission) and for the ranking of small calls with the
general emission and tile sort.
"""
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2505_18992_gb300 import build as B
from paper_2505_18992_gb300 import scenes
from tests.helpers import assert_grad_close, masked_upstream

pytestmark = pytest.mark.gpu

NAMES = ("means", "scales", "quats", "opacities", "colors")

# run in the variant's process: renders the scenes, two backwards of the first
CHILD = """
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
from paper_2505_18992_gb300 import build
build.build()
from paper_2505_18992_gb300.render import Intrinsics, Renderer
d = np.load(sys.argv[2])
res = {}
for s in ("tile", "frame", "rank"):
    t = lambda k, dt=torch.float32: torch.as_tensor(d[s + "_" + k], dtype=dt, device="cuda")
    W, H, fx, fy, cx, cy = d[s + "_cam"]
    r = Renderer(Intrinsics(int(W), int(H), fx, fy, cx, cy), tile_w=16, tile_h=int(d[s + "_tile_h"]))
    names = ("means", "scales", "quats", "opacities", "colors")
    g, T = [t(k) for k in names], t("T", torch.float64)
    out = r.forward(*g, T)
    res.update({s + "_" + k: v.cpu().numpy() for k, v in out.items()})
    if s == "tile":
        for form in ("full", "geometric"):
            grads = {k: torch.zeros_like(x) for k, x in zip(names, g) if form == "full" or k in names[:3]}
            r.backward(*g, T, out, t("up0"), t("up1"), t("up2"), grads=grads, check=True)
            res.update({form + "_" + k: v.cpu().numpy() for k, v in grads.items()})
np.savez(sys.argv[3], **res)
"""


def _inputs():
    tile = scenes.random_gaussians(60, 16, 4, 20.0, 3, scale_range=(0.02, 0.5))
    frame = scenes.random_gaussians(20_000, 320, 240, 300.0, 4, scale_range=(0.005, 0.05))
    rank = scenes.random_gaussians(6_000, 800, 900, 700.0, 5, scale_range=(0.005, 0.05))
    ref = oracle.render_scene(tile)
    up = masked_upstream(scenes.upstream_grads(5, 1, 4, 16), ref["flags"])
    d = {}
    for s, sc, h in (("tile", tile, 4), ("frame", frame, 16), ("rank", rank, 16)):
        c = sc.camera
        d.update({s + "_" + k: a for k, a in zip(NAMES, sc.arrays())})
        d.update({s + "_T": c.T_cw, s + "_tile_h": h, s + "_cam": [c.width, c.height, c.fx, c.fy, c.cx, c.cy]})
    d.update({"tile_up%d" % i: u for i, u in enumerate(up)})
    return d, oracle.render_scene(tile, grads=up)


def _run(root, tmp, inputs, flags):
    env = {**os.environ, "VPGS_NVCC_FLAGS": flags}
    np.savez(tmp / "in.npz", **inputs)
    res = subprocess.run([sys.executable, "-c", CHILD, str(root), str(tmp / "in.npz"), str(tmp / "out.npz")],
                         env=env, cwd=str(root), capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stderr[-2000:]
    return np.load(tmp / "out.npz")


@pytest.fixture(scope="module")
def case(tmp_path_factory):
    inputs, ref = _inputs()
    return inputs, ref, _run(B.ROOT, tmp_path_factory.mktemp("default"), inputs, "")


def _variant(case, tmp_path, flags):
    root = tmp_path / "tree"
    shutil.copytree(B.PKG, root / "paper_2505_18992_gb300",
                    ignore=shutil.ignore_patterns("_build", "*.so", "__pycache__"))
    shutil.copytree(os.path.join(B.ROOT, "include"), root / "include")
    return _run(root, tmp_path, case[0], flags)


def test_ieee_divisions_reach_the_main_walk(case, tmp_path):
    _, ref, base = case
    got = _variant(case, tmp_path, "-DVPGS_BWD_RCP=0")
    for form in ("full", "geometric"):
        names = NAMES if form == "full" else NAMES[:3]
        for k in names:
            assert_grad_close(got[f"{form}_{k}"], ref["d_" + k], k)
        # T recovered by divisions: other last bits than by reciprocals
        assert any(not np.array_equal(got[f"{form}_{k}"], base[f"{form}_{k}"]) for k in names), form


@pytest.mark.parametrize("flags", ["-DVPGS_DEPTH_SORT_ITEMS=8 -DVPGS_TILE_SORT_ITEMS=8",
                                   "-DVPGS_DEPTH_SORT_ITEMS=16 -DVPGS_TILE_SORT_ITEMS=32"])
def test_sort_widths_give_the_same_lists(case, tmp_path, flags):
    got = _variant(case, tmp_path, flags)
    for k in ("rgb", "depth", "alpha", "t_final", "n_contrib", "n_iter"):
        for s in ("frame", "rank"):
            assert np.array_equal(got[f"{s}_{k}"], case[2][f"{s}_{k}"]), (s, k)
