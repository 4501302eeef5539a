"""With one view per surfel the preprocess drops surfels from center and size
alone where it can; whatever it is given, its records are those of the general
path (two views per surfel) bit for bit: surfels all around the frustum, near,
far and behind, small and as large as their distance, maps far from the
origin, rotations with a scale and a shear, unusable surfels, either tile
shape, with and without the low-pass extent."""
import numpy as np
import pytest
import torch

from paper_2604_03092_gb300 import scenes
from paper_2604_03092_gb300.rasterizer import RasterConfig, Rasterizer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile,lowpass", [(8, 0.70710678), (16, 0.0), (8, 6.0)])
@pytest.mark.parametrize("scales,origin,stretch", [((0.001, 0.05), 0.0, 1.0), ((0.05, 8.0), 0.0, 1.0),
                                                   ((0.01, 0.5), 3000.0, 1.0), ((0.01, 0.5), 0.0, 2.5)])
def test_records_equal_general_path(tile, lowpass, scales, origin, stretch):
    n, w, h = 30_000, 203, 149
    rng = np.random.default_rng(int(tile + 10 * scales[1] + origin + 100 * stretch))
    sc = scenes.random_scene(n=n, width=w, height=h, f=170.0, seed=3, depth_range=(-6.0, 14.0), xy_range=9.0,
                             scale_range=scales)
    rot, _ = np.linalg.qr(rng.normal(size=(3, 3)))
    rot *= np.sign(np.linalg.det(rot))
    t = rng.normal(size=3)
    world = (sc.means - t) @ rot + origin * np.array([1.0, -0.5, 0.25])  # camera = rot (world - shift) + t
    shear = np.eye(3) * stretch
    shear[0, 1] = 0.3 * (stretch - 1.0)
    rt = np.concatenate([shear @ rot, (shear @ (t - rot @ (origin * np.array([1.0, -0.5, 0.25]))))[:, None]], 1)
    means, scale, quats = world.astype(np.float32), sc.scales.copy(), sc.quats.copy()
    opacity = sc.opacity.copy()
    means[::97, 1], quats[5::101], opacity[7::53], scale[11::103] = np.nan, 0.0, 0.001, 0.0
    scale[13::107] *= -1.0
    view = scenes.View(w, h, 170.0, 165.0, 90.0, 80.0, rt.astype(np.float32))
    prm = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (means, scale, quats, opacity, sc.rgb)]
    cfg = RasterConfig(tile_w=tile, tile_h=tile, lowpass_sigma=lowpass)
    got = []
    for k in (1, 2):
        rast = Rasterizer([view] * k, n, cfg, capacity=64)  # only the preprocess runs
        rast.preprocess(*prm)
        nt = rast.ws_tensor(rast.layout.ntiles, n, torch.int32).clone()
        rec = rast.ws_tensor(rast.layout.records, 20 * n, torch.int32).view(n, 20).clone()
        got.append((nt, rec, rast.stats()["n_visible"] / k))
    (nt1, rec1, vis1), (nt2, rec2, vis2) = got
    assert torch.equal(nt1, nt2) and vis1 == vis2
    inside = nt1 != 0
    assert 100 < int(inside.sum()) < 0.7 * n
    assert torch.equal(rec1[inside], rec2[inside])
