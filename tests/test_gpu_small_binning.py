"""The binning's forms for small calls against its general forms.

Small calls rank their visible (view, Gaussian) pairs by comparison (up to 6,144
pairs) and, up to 12,288 pairs and 15M pairs x tiles, every tile selects its list
from them; 257 to 512 tiles otherwise take one sort pass of 9-bit digits.  All are exact reorderings, so a
call padded past a limit with invisible Gaussians, or rendered with tiles of
another shape, gives the same images.
"""
import numpy as np
import pytest
import torch

from paper_2505_18992_gb300 import scenes
from paper_2505_18992_gb300.render import Intrinsics, Renderer
from tests.helpers import dev

pytestmark = pytest.mark.gpu


def _render(arrays, cam, **opts):
    r = Renderer(Intrinsics(cam.width, cam.height, cam.fx, cam.fy, cam.cx, cam.cy), n_views=cam.n_views, **opts)
    out = r.forward(*[dev(a) for a in arrays], dev(cam.T_cw, torch.float64), check=True)
    st = r.stats()
    return {k: v.cpu().numpy() for k, v in out.items()}, (st.n_visible, st.n_instances)


@pytest.mark.parametrize("views,n,size,scale", [
    (1, 1, (120, 90), 0.02), (1, 31, (120, 90), 0.02), (1, 33, (120, 90), 0.6), (1, 1024, (120, 90), 0.02),
    (1, 1025, (333, 600), 0.6), (1, 8193, (120, 90), 0.02), (1, 12288, (120, 90), 0.02), (3, 4096, (97, 61), 0.1),
    (3, 2048, (700, 640), 0.3), (1, 6145, (700, 900), 0.02),  # past 15M pairs x tiles: by rank, general
    # emission: Gaussians of many tile rows, in chunks that hold them as runs and that do not
    (1, 500, (1900, 1000), 0.5), (1, 300, (400, 4000), 1.5),
    (1, 900, (4120, 20), 0.05), (1, 900, (20, 4120), 0.05)])  # more than 256 columns or rows of tiles
def test_small_forms_equal_the_general_ones(views, n, size, scale):
    sc = scenes.random_gaussians(n, *size, 1.1 * max(size), seed=n, scale_range=(0.005, scale), n_views=views)
    if n > 8:
        sc.means[n // 2:n // 2 + 4] = sc.means[0]  # equal depths go by index
    sc.opacities[::7] = 0.001                    # culled ones in between
    a, na = _render(sc.arrays(), sc.camera)
    pad = 20_000 - n  # past the limit: the same Gaussians, then invisible ones
    arrays = [np.concatenate([x, np.repeat(x[:1], pad, 0)]) for x in sc.arrays()]
    arrays[3][n:] = 0.0
    b, nb = _render(arrays, sc.camera)
    assert na == nb
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def test_small_call_reports_too_many_instances():
    sc = scenes.random_gaussians(500, 120, 90, 130.0, seed=1, scale_range=(0.05, 0.2))
    cam = sc.camera
    r = Renderer(Intrinsics(cam.width, cam.height, cam.fx, cam.fy, cam.cx, cam.cy))
    r.reserve(500, max_instances=64)
    g, T = [dev(a) for a in sc.arrays()], dev(cam.T_cw, torch.float64)
    r.forward(*g, T, check=False)
    st = r.stats()
    assert st.status == 2 and st.n_instances > 64
    out = r.forward(*g, T, check=True)  # grows and renders
    want, _ = _render(sc.arrays(), cam)
    assert np.array_equal(out["rgb"].cpu().numpy(), want["rgb"])


@pytest.mark.parametrize("tiles", [(16, 16), (257, 1), (17, 16), (32, 16), (27, 19)])
def test_nine_bit_tile_pass(tiles):
    W, H = 16 * tiles[0] - 3, 16 * tiles[1] - 5
    sc = scenes.random_gaussians(3000, W, H, 0.8 * max(W, H), seed=tiles[0], scale_range=(0.002, 0.03))
    a, _ = _render(sc.arrays(), sc.camera)
    b, _ = _render(sc.arrays(), sc.camera, tile_w=8, tile_h=8)
    assert np.array_equal(a["n_contrib"], b["n_contrib"])
    for k in ("rgb", "depth", "alpha", "t_final"):
        assert np.abs(a[k] - b[k]).max() <= 1e-5, k
