"""Instance overflow in each form of the binning: reported by status and count, with
nothing written outside the workspace and the images, right up to the exact capacity."""
import numpy as np
import pytest
import torch

from paper_2505_18992_gb300 import scenes
from paper_2505_18992_gb300.render import Intrinsics, Renderer
from tests.helpers import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,size", [(300_000, (640, 480)),   # general: scans, sorts, emission by many blocks
                                    (6_000, (800, 900)),     # small by rank, general emission
                                    (5_000, (320, 240))])    # small by rank and tile lists
def test_overflow_is_reported_and_stays_inside(n, size):
    sc = scenes.random_gaussians(n, *size, 0.8 * size[0], seed=n, scale_range=(0.005, 0.02))
    cam = sc.camera
    g, T = [dev(a) for a in sc.arrays()], dev(cam.T_cw, torch.float64)
    intr = Intrinsics(cam.width, cam.height, cam.fx, cam.fy, cam.cx, cam.cy)
    full = Renderer(intr)
    want = {k: v.cpu().numpy() for k, v in full.forward(*g, T).items()}
    total = full.last_stats.n_instances
    guard = 1 << 16
    for cap in (64, total // 2, total - 256, total):  # (a workspace holds up to 63 more than it was asked for)
        r = Renderer(intr)
        r.reserve(n, max_instances=cap)
        ws = torch.full((r.ws_bytes + guard,), 0xA5, dtype=torch.uint8, device="cuda")
        r.ws = ws[:r.ws_bytes]  # same base address, so still 16-byte aligned
        out = r.alloc_images()
        for _ in range(5):
            r.forward(*g, T, out=out, check=False)
            st = r.stats()
            assert (st.status, st.n_instances) == (0 if cap == total else 2, total)
        assert bool((ws[r.ws_bytes:] == 0xA5).all())
        if cap < total:
            r.forward(*g, T, out=out, check=True)  # grows and renders
        for k in want:
            assert np.array_equal(out[k].cpu().numpy(), want[k]), (cap, k)
