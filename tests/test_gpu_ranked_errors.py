"""Attributed errors on 8x8 tiles (pixels ranked by error, masks transposed)
against the kernel of the 256-pixel tiles, over the forms of the error map:
ties, zeros, negative, NaN and infinite errors, tiles cut by the image, lists
around a 32-entry word, and raised into what the caller holds."""
import numpy as np
import pytest
import torch

from gpu_utils import gpu_forward
from paper_2604_03092_gb300 import scenes
from paper_2604_03092_gb300.rasterizer import RasterConfig

pytestmark = pytest.mark.gpu


def _errors(kind, n, rng):
    e = rng.uniform(0.1, 2.0, n).astype(np.float32)
    if kind == "ties":
        e = np.round(e * 2).astype(np.float32) / 2
    elif kind == "sparse":
        e[rng.uniform(size=n) < 0.9] = 0.0
    elif kind == "odd":
        e[::5], e[1::7], e[2::11], e[3::13] = -1.0, np.nan, np.inf, -0.0
    elif kind == "zero":
        e[:] = 0.0
    return e


@pytest.mark.parametrize("kind", ["random", "ties", "sparse", "odd", "zero"])
@pytest.mark.parametrize("n,width,height", [(1, 8, 8), (33, 9, 5), (64, 24, 20), (700, 130, 67)])
def test_equal_on_both_tile_shapes(kind, n, width, height):
    """16x16 tiles take the pairs one by one; both shapes blend the same pairs but for surfels within rounding
    of a threshold, and the scenes' pair counts say that there is none."""
    sc = scenes.random_scene(n=n, width=width, height=height, f=float(max(width, height)), seed=n,
                             scale_range=(0.05, 0.6))
    sc.opacity = np.clip(sc.opacity, 0.01, 0.6).astype(np.float32)
    err = torch.from_numpy(_errors(kind, width * height, np.random.default_rng(n))).cuda()
    held = torch.rand(n, device="cuda")
    got, blended = [], []
    for tile in (8, 16):
        rast, _, _ = gpu_forward(sc, RasterConfig(tile_w=tile, tile_h=tile))
        got.append((rast.max_error(err), rast.max_error(err, held.clone())))
        blended.append(rast.stats()["fwd_pairs_blended"])
    assert blended[0] == blended[1]
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert torch.equal(got[0][1], torch.maximum(got[0][0], held))
