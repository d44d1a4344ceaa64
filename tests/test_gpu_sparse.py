"""Calls most of whose tiles are empty: their blocks leave early, with one tile per block
and with blocks that pull tiles from a queue, and the other tiles are unaffected."""
import numpy as np
import pytest
import torch

import oracle
from oracle.raster import Options
from paper_2505_18992_gb300 import scenes
from paper_2505_18992_gb300.render import Intrinsics, Renderer
from tests.helpers import assert_grad_close, assert_images_close, assert_pose_close, dev, masked_upstream

pytestmark = pytest.mark.gpu

NAMES = ("means", "scales", "quats", "opacities", "colors")


@pytest.mark.parametrize("geometric", [False, True])
@pytest.mark.parametrize("persistent", [0, 1])
@pytest.mark.parametrize("n,size,tile", [(1, (640, 480), (16, 16)), (5, (201, 119), (16, 16)),
                                         (5, (201, 119), (32, 2)), (5, (201, 119), (4, 64)), (40, (1000, 700), (8, 8))])
def test_mostly_empty_tiles(n, size, tile, persistent, geometric):
    sc = scenes.random_gaussians(n, *size, 0.9 * size[0], seed=n, scale_range=(0.005, 0.03))
    bg = (0.2, 0.4, 0.6)
    opts = Options(bg=bg, tile_w=tile[0], tile_h=tile[1])
    ref0 = oracle.render_scene(sc, opts=opts)
    up = masked_upstream(scenes.upstream_grads(n, 1, size[1], size[0]), ref0["flags"])
    ref = oracle.render_scene(sc, grads=up, opts=opts)
    cam = sc.camera
    r = Renderer(Intrinsics(*size, cam.fx, cam.fy, cam.cx, cam.cy), tile_w=tile[0], tile_h=tile[1], bg=bg,
                 persistent_ctas=persistent)
    g, T = [dev(a) for a in sc.arrays()], dev(cam.T_cw, torch.float64)
    out = r.forward(*g, T, check=True)
    got = {k: v.cpu().numpy() for k, v in out.items()}
    assert_images_close(got, ref0, ref0["flags"])
    empty = got["n_contrib"] == 0
    assert empty.mean() > 0.5 and (got["t_final"][empty] == 1.0).all()
    names = NAMES[:3] if geometric else NAMES
    grads = {k: torch.zeros_like(t) for k, t in zip(names, g)}
    dpose = torch.zeros((1, 6), dtype=torch.float64, device="cuda")
    r.backward(*g, T, out, *[dev(u) for u in up], grads=grads, dpose=dpose, check=True)
    for k in names:
        assert_grad_close(grads[k].cpu().numpy(), ref["d_" + k], k)
    assert_pose_close(dpose.cpu().numpy(), ref["d_pose"])
