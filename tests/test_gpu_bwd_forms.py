"""The compositing backward's two-phase form at the sizes where it can go wrong, and
the values that must not leak through its masked lanes.

The kernel collects list entries in groups of 8 from batches of one record per
thread, and lanes that do not blend take part with alpha = 0.  Tolerances: the
parity rules of tests/helpers.py against the FP64 oracle; between two renders of
the same kernel only the order of float32 atomics differs, a few ulps of the
summed magnitudes, bounded here by 1e-4 of a tensor's rms.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2505_18992_gb300 import scenes
from paper_2505_18992_gb300.render import Intrinsics, Renderer
from tests.helpers import assert_grad_close, dev, masked_upstream

pytestmark = pytest.mark.gpu

NAMES = ("means", "scales", "quats", "opacities", "colors")


def _scene(n, W, H, seed, opac):
    """n Gaussians that each cover most of the image, thin enough that all of them blend."""
    sc = scenes.random_gaussians(n, W, H, 40.0, seed, depth=(2.0, 3.0), spread=0.5, scale_range=(0.3, 0.6))
    sc.opacities = np.random.default_rng(seed).uniform(*opac, size=n).astype(np.float32)
    return sc


def _render(sc, tile, up, **opts):
    cam = sc.camera
    r = Renderer(Intrinsics(cam.width, cam.height, cam.fx, cam.fy, cam.cx, cam.cy), n_views=cam.n_views,
                 tile_w=tile[0], tile_h=tile[1], **opts)
    g, T = [dev(a) for a in sc.arrays()], dev(cam.T_cw, torch.float64)
    out = r.forward(*g, T, check=True)
    up = [None if u is None else dev(u) for u in up(out)]
    grads = {k: torch.zeros_like(t) for k, t in zip(NAMES, g)}
    r.backward(*g, T, out, *up, grads=grads, check=True)
    return out, {k: v.cpu().numpy() for k, v in grads.items()}


@pytest.mark.parametrize("tile", [(16, 16), (4, 16), (32, 16)])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 63, 64, 65, 129, 257])
def test_group_and_batch_edges(n, tile):
    sc = _scene(n, 37, 21, seed=n, opac=(0.01, 0.03))
    ref0 = oracle.render_scene(sc)
    up = masked_upstream(scenes.upstream_grads(n, 1, 21, 37), ref0["flags"])
    ref = oracle.render_scene(sc, grads=up)
    _, grads = _render(sc, tile, lambda out: up)
    for k in NAMES:
        assert_grad_close(grads[k], ref["d_" + k], k)


def _same(a, b, rows, name):
    rms = np.sqrt(np.mean(np.square(b[rows], dtype=np.float64)))
    assert np.isfinite(a[rows]).all(), name
    assert np.abs(a[rows] - b[rows]).max() <= 1e-4 * rms, name


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 3e37])
def test_upstream_of_one_pixel_stays_with_the_gaussians_that_blend_there(value):
    sc = scenes.random_gaussians(300, 64, 48, 70.0, seed=5)
    rng = np.random.default_rng(3)
    g = rng.normal(size=(1, 3, 48, 64)).astype(np.float32)

    def at(x):
        u = g.copy()
        u[0, :, 20, 30] = x
        return u

    hot = np.zeros_like(g)
    hot[0, :, 20, 30] = 1.0
    _, one = _render(sc, (16, 16), lambda out: (hot, None, None))
    here = np.abs(one["colors"]).max(1) > 0  # the Gaussians that blend into the pixel
    assert 0 < here.sum() < 150
    _, want = _render(sc, (16, 16), lambda out: (at(0.0), None, None))
    _, got = _render(sc, (16, 16), lambda out: (at(value), None, None))
    for k in NAMES:
        _same(got[k], want[k], ~here, k)


def test_a_huge_colour_stays_with_its_pixels():
    sc = scenes.random_gaussians(300, 64, 48, 70.0, seed=6)
    rng = np.random.default_rng(4)
    g = 100.0 * rng.normal(size=(1, 3, 48, 64)).astype(np.float32)
    near = int(np.argmin(sc.means[:, 2]))  # in front: what it covers is known from the image
    sc.opacities[near] = 0.6
    sc.colors[near] = 0.0
    base = sc.colors.copy()
    sc.colors[near] = 1e6
    marked, _ = _render(sc, (16, 16), lambda out: (g, None, None))
    seen = (marked["rgb"].amax(1) > 100.0).cpu().numpy()[0]
    assert 0 < seen.sum() < 2000
    up = np.where(seen[None, None], 0.0, g).astype(np.float32)
    sc.colors[near] = 1e38  # (the three channels of a record must sum to a finite value)
    _, got = _render(sc, (16, 16), lambda out: (up, None, None))
    sc.colors = base
    _, want = _render(sc, (16, 16), lambda out: (up, None, None))
    for k in NAMES:
        _same(got[k], want[k], slice(None), k)
