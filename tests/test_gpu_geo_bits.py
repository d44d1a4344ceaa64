"""The geometric compositing backward's sums, bit for bit.

tests/golden/geometric_backward_bits.json holds digests of the gradients and pose
gradients that the branching kernel gave before the masked walk replaced it (GB300, the
default build) for scenes of one tile and one warp, where every sum has a single order.
A pose tracker feeds on these roundings, so the values are pinned and not only their
accuracy; `python tests/test_gpu_geo_bits.py` prints the digests of the tree it runs in.
"""
import hashlib
import json
import os

import pytest
import torch

from paper_2505_18992_gb300 import scenes
from paper_2505_18992_gb300.render import Intrinsics, Renderer

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "geometric_backward_bits.json")
NAMES = ("means", "scales", "quats")
TILES = ((16, 4), (4, 16), (8, 8), (32, 2))


def _digests(tile, n, seed):
    W, H = tile
    sc = scenes.random_gaussians(n, W, H, 20.0, seed, scale_range=(0.02, 0.5))
    if seed % 3 == 2:
        sc.scales[::5, 1:] = 1e-4  # needles: the double-float evaluation
    if seed % 4 == 3:
        sc.opacities *= 0.1        # long lists
    g = [torch.tensor(a, device="cuda") for a in sc.arrays()]
    T = torch.tensor(sc.camera.T_cw, device="cuda")
    r = Renderer(Intrinsics(W, H, 20.0, 20.0, W / 2.0, H / 2.0), tile_w=W, tile_h=H)
    out = r.forward(*g, T, check=True)
    up = [torch.tensor(u, device="cuda") for u in scenes.upstream_grads(seed, 1, H, W)]
    got = {k: torch.zeros_like(t) for k, t in zip(NAMES, g)}
    pose = torch.zeros((1, 6), dtype=torch.float64, device="cuda")
    r.backward(*g, T, out, *up, grads=got, dpose=pose, check=True)
    got["pose"] = pose
    # (+ 0: a sum of zeros has no sign worth pinning)
    return {k: hashlib.sha256((v.cpu().numpy() + 0.0).tobytes()).hexdigest()[:16] for k, v in got.items()}


def _cases():
    return [(tile, n, seed) for i, tile in enumerate(TILES) for j, n in enumerate((1, 3, 40, 64, 65, 200))
            for seed in (10 * i + j,)]


def _name(tile, n, seed):
    return "%dx%d %d %d" % (*tile, n, seed)


@pytest.mark.parametrize("tile,n,seed", _cases(), ids=lambda v: str(v))
def test_bits(tile, n, seed):
    with open(GOLDEN) as f:
        want = json.load(f)[_name(tile, n, seed)]
    assert _digests(tile, n, seed) == want


if __name__ == "__main__":
    print(json.dumps({_name(*c): _digests(*c) for c in _cases()}, indent=0))
