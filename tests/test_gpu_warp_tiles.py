"""8x8 tiles are composited by a warp per tile, or per half tile where there
are few: sizes at the edges of that design (images smaller than a tile, lists
around one 32-entry chunk, chunks whose pairs overflow the backward's slots
or take the forward's dense walk, enough tiles for whole ones), forward and
gradients against the FP64 oracle within the library's parity bar."""
import numpy as np
import pytest
import torch

import oracle
from gpu_utils import FWD_ATOL, GRAD_REL_L2, gpu_forward, oracle_cfg, rel_l2, unresolved_flagged, upstream, view_stack
from paper_2604_03092_gb300 import scenes
from paper_2604_03092_gb300.rasterizer import RasterConfig

pytestmark = pytest.mark.gpu

SMALL, WIDE = (0.02, 0.3), (0.6, 1.5)  # scales: a few pixels, every pixel of the image


@pytest.mark.parametrize("n,width,height,scales,opacity,ray", [
    (1, 1, 1, WIDE, 0.9, False),
    (31, 7, 3, SMALL, 0.5, False),
    (32, 8, 8, WIDE, 0.1, True),
    (33, 9, 5, WIDE, 0.3, False),
    (65, 17, 33, SMALL, 0.5, True),
    (200, 24, 20, WIDE, 0.05, False),   # 2048 pairs per chunk, tiles saturate after several chunks
    (97, 40, 24, (0.05, 1.0), 0.3, True),
    (300, 648, 520, (0.3, 0.8), 0.08, True),  # 5265 tiles: one warp per whole tile
])
def test_forward_and_gradients_match_oracle(n, width, height, scales, opacity, ray):
    sc = scenes.random_scene(n=n, width=width, height=height, f=max(0.8 * max(width, height), 4.0), seed=n,
                             scale_range=scales)
    sc.opacity = np.clip(sc.opacity * 2 * opacity, 0.01, 0.99).astype(np.float32)
    cfg = RasterConfig(bg=(0.2, 0.1, 0.3), depth_ray=ray)
    rast, params, im = gpu_forward(sc, cfg)
    d_dev, d_views = upstream(rast, 5)
    grads = rast.backward(*params, d_dev)
    torch.cuda.synchronize()
    st = rast.stats()
    assert st["status"] == 0 and st["bwd_pairs_blended"] == st["fwd_pairs_blended"]
    p = oracle.preprocess_scene_view(sc, 0, oracle_cfg(cfg))
    ref = oracle.render(p)
    gpu = view_stack(rast, im, 0)
    near = (ref.pflags & (oracle.PF_FORWARD | (oracle.PF_BRANCH if ray else 0))) != 0
    if (~near).any():
        assert np.abs(gpu - ref.out)[:, ~near].max() <= FWD_ATOL
    flagged = np.flatnonzero((ref.pflags & oracle.PF_FORWARD).reshape(-1))
    assert unresolved_flagged(gpu.reshape(8, -1)[:, flagged], p, flagged) <= 1e-4 * near.size + (1 if ray else 0)
    og = oracle.render_bwd(sc.means, sc.scales, sc.quats, p, d_views[0])
    for name in ("means", "scales", "quats", "opacity", "rgb"):
        assert rel_l2(getattr(grads, name).cpu().numpy(), getattr(og, name)) <= GRAD_REL_L2, name
    assert rel_l2(grads.pose.cpu().numpy()[0], og.pose) <= GRAD_REL_L2
