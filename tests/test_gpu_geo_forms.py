"""The geometric compositing backward (no opacity or colour gradient asked, as in pose
tracking) at the sizes where it can go wrong, and against the branching walk.

It takes list entries two at a time from batches of two records per thread, lanes that
do not blend take part with alpha = 0, and each entry's six sums go through a warp
reduction or, for one or two blending lanes, their own atomics.  Tolerances: the parity
rules of tests/helpers.py against the FP64 oracle; where a tile is one warp every sum has
one order, and the masked walk gives the branching walk's bits.
"""
import numpy as np
import pytest
import torch

import oracle
from oracle.raster import Options
from paper_2505_18992_gb300 import scenes
from paper_2505_18992_gb300.render import Intrinsics, Renderer
from tests.helpers import assert_grad_close, assert_pose_close, dev, masked_upstream

pytestmark = pytest.mark.gpu

NAMES = ("means", "scales", "quats")


def _render(sc, tile, up, **opts):
    """Forward and geometric backward: images, gradients and the pose gradient."""
    cam = sc.camera
    r = Renderer(Intrinsics(cam.width, cam.height, cam.fx, cam.fy, cam.cx, cam.cy), tile_w=tile[0], tile_h=tile[1],
                 **opts)
    g, T = [dev(a) for a in sc.arrays()], dev(cam.T_cw, torch.float64)
    out = r.forward(*g, T, check=True)
    grads = {k: torch.zeros_like(t) for k, t in zip(NAMES, g)}
    dpose = torch.zeros((1, 6), dtype=torch.float64, device="cuda")
    r.backward(*g, T, out, *[None if u is None else dev(u) for u in up], grads=grads, dpose=dpose, check=True)
    return out, {k: v.cpu().numpy() for k, v in grads.items()}, dpose.cpu().numpy(), r.last_stats.n_instances


# 128 threads stage 256 records a batch, 32 threads 64, 256 threads 512
@pytest.mark.parametrize("tile,n", [((16, 16), n) for n in (1, 2, 3, 255, 256, 257, 511, 512, 513)] +
                                   [((4, 16), n) for n in (1, 2, 3, 63, 64, 65, 127, 128, 129)] +
                                   [((32, 16), n) for n in (511, 512, 513)])
def test_walk_and_batch_edges(tile, n):
    # one ragged tile that every Gaussian covers, thin enough that all of them blend
    W, H = tile[0] - 1, tile[1] - 1
    sc = scenes.random_gaussians(n, W, H, 40.0, seed=n, depth=(2.0, 3.0), spread=0.5, scale_range=(0.6, 1.0))
    sc.opacities = np.random.default_rng(n).uniform(0.006, 0.010, size=n).astype(np.float32)
    opts = Options(alpha_min=1e-3, tile_w=tile[0], tile_h=tile[1])
    ref0 = oracle.render_scene(sc, opts=opts)
    up = masked_upstream(scenes.upstream_grads(n, 1, H, W), ref0["flags"])
    ref = oracle.render_scene(sc, grads=up, opts=opts)
    out, grads, dpose, listed = _render(sc, tile, up, alpha_min=1e-3)
    assert listed == n and int(out["n_iter"].max()) == n
    for k in NAMES:
        assert_grad_close(grads[k], ref["d_" + k], k)
    assert_pose_close(dpose, ref["d_pose"])


@pytest.mark.parametrize("n", [1, 2, 3, 31, 62, 63, 64, 65, 127, 128, 129, 200])
def test_masked_walk_gives_the_branching_walks_bits(n):
    # a farthest Gaussian over the first column's top, where no gradient arrives: its colour
    # changes no gradient, but a huge one sends every batch to the branching walk
    sc = scenes.random_gaussians(n, 4, 16, 20.0, seed=100 + n, spread=0.5, scale_range=(0.3, 0.8))
    sc.opacities = np.random.default_rng(n).uniform(0.008, 0.02, size=n).astype(np.float32)  # it stays visible
    sc.opacities[0] = 1.0  # one whose alpha is clamped near its centre
    for k, row in (("means", [-1.5 * 6.0 / 20.0, -6.0 * 6.0 / 20.0, 6.0]), ("scales", [0.1] * 3),
                   ("quats", [1.0, 0.0, 0.0, 0.0]), ("opacities", 0.5), ("colors", [0.5] * 3)):
        setattr(sc, k, np.concatenate([getattr(sc, k), np.asarray(row, np.float32)[None]]))
    up = [np.array(u) for u in scenes.upstream_grads(n, 1, 16, 4)]
    for u in up:
        u[..., :6, :] = 0.0
    _, plain, plain_pose, _ = _render(sc, (4, 16), up)
    sc.colors[-1] = 1e16
    out, branching, branching_pose, listed = _render(sc, (4, 16), up)
    seen = (out["rgb"][0].abs().amax(0) > 1e10).cpu().numpy()
    assert listed == n + 1 and seen[:6].any() and not seen[6:].any()
    for k in NAMES:
        assert np.isfinite(plain[k]).all()
        assert np.array_equal(plain[k], branching[k]), k
    assert np.array_equal(plain_pose, branching_pose)


def _same(a, b, rows, name):
    # only the order of float32 atomics differs: a few ulps of the summed magnitudes
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

    # the Gaussians that blend into the pixel: those that a gradient arriving only there reaches
    hot = np.zeros_like(g)
    hot[0, :, 20, 30] = (1.0, -0.5, 0.25)
    _, one, _, _ = _render(sc, (16, 16), (hot, None, None))
    here = np.abs(one["means"]).max(1) > 0
    assert 0 < here.sum() < 150
    _, want, _, _ = _render(sc, (16, 16), (at(0.0), None, None))
    _, got, _, _ = _render(sc, (16, 16), (at(value), None, None))
    for k in NAMES:
        _same(got[k], want[k], ~here, k)


def test_a_huge_colour_stays_with_its_pixels():
    sc = scenes.random_gaussians(300, 64, 48, 70.0, seed=6)
    g = 100.0 * np.random.default_rng(4).normal(size=(1, 3, 48, 64)).astype(np.float32)
    near = int(np.argmin(sc.means[:, 2]))  # in front: what it covers is known from the image
    sc.opacities[near] = 0.6
    sc.colors[near] = 0.0
    base = sc.colors.copy()
    sc.colors[near] = 1e6
    marked, _, _, _ = _render(sc, (16, 16), (g, None, None))
    seen = (marked["rgb"].amax(1) > 100.0).cpu().numpy()[0]
    assert 0 < seen.sum() < 2000
    up = np.where(seen[None, None], 0.0, g).astype(np.float32)
    sc.colors[near] = 1e38  # (the three channels of a record must sum to a finite value)
    _, got, got_pose, _ = _render(sc, (16, 16), (up, None, None))
    sc.colors = base
    _, want, want_pose, _ = _render(sc, (16, 16), (up, None, None))
    for k in NAMES:
        _same(got[k], want[k], slice(None), k)
    assert np.abs(got_pose - want_pose).max() <= 1e-4 * np.abs(want_pose).max()
