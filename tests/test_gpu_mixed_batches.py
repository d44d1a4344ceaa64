"""The compositing backward on lists that mix near-degenerate records, which add their sums
entry by entry, with plain ones, which are summed eight at a time (full form) or two at a
time (geometric form), against the FP64 oracle by the parity rules of tests/helpers.py."""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_18992_gb300 import scenes
from paper_2505_18992_gb300.render import Intrinsics, Renderer
from tests.helpers import assert_grad_close, assert_images_close, assert_pose_close, dev, masked_upstream

pytestmark = pytest.mark.gpu

NAMES = ("means", "scales", "quats", "opacities", "colors")


@pytest.mark.parametrize("geometric", [False, True])
@pytest.mark.parametrize("every", [1, 2, 9])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 64, 129, 257])
def test_near_degenerate_entries_between_plain_ones(n, every, geometric):
    W, H = 37, 21
    sc = scenes.random_gaussians(n, W, H, 40.0, seed=n, depth=(2.0, 3.0), spread=0.5, scale_range=(0.3, 0.6))
    sc.opacities = np.random.default_rng(n).uniform(0.01, 0.03, size=n).astype(np.float32)
    sc.scales[::every] = (1.0, 1e-4, 1e-4)  # needles: condition numbers of several hundred
    ref0 = oracle.render_scene(sc)
    up = masked_upstream(scenes.upstream_grads(n, 1, H, W), ref0["flags"])
    ref = oracle.render_scene(sc, grads=up)
    cam = sc.camera
    r = Renderer(Intrinsics(W, H, cam.fx, cam.fy, cam.cx, cam.cy))
    g, T = [dev(a) for a in sc.arrays()], dev(cam.T_cw, torch.float64)
    out = r.forward(*g, T, check=True)
    assert_images_close({k: v.cpu().numpy() for k, v in out.items()}, ref0, ref0["flags"])
    names = NAMES[:3] if geometric else NAMES
    grads = {k: torch.zeros_like(t) for k, t in zip(names, g)}
    dpose = torch.zeros((1, 6), dtype=torch.float64, device="cuda")
    r.backward(*g, T, out, *[dev(u) for u in up], grads=grads, dpose=dpose, check=True)
    for k in names:
        assert_grad_close(grads[k].cpu().numpy(), ref["d_" + k], k)
    assert_pose_close(dpose.cpu().numpy(), ref["d_pose"])
