"""8x8 tiles with few pixels still compositing at the start of a chunk are
handed from the warp-per-tile forward to the kernel of the tails: handed over
never, at once or on the way, at each chunk size, lists that end within and
at the edge of a chunk, tiles cut by the image, halves and whole tiles;
forward and gradients against the FP64 oracle within the library's parity
bar."""
import numpy as np
import pytest
import torch

import oracle
from gpu_utils import FWD_ATOL, GRAD_REL_L2, gpu_forward, oracle_cfg, rel_l2, unresolved_flagged, upstream, view_stack
from paper_2604_03092_gb300 import scenes
from paper_2604_03092_gb300.rasterizer import RasterConfig

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,width,height,chunk,tail,ray", [
    (1, 1, 1, 64, 255, False),
    (64, 9, 5, 64, 255, True),
    (65, 40, 24, 64, 3, False),
    (700, 40, 24, 64, 20, True),
    (256, 17, 33, 128, 255, False),
    (900, 24, 20, 128, 0, False),
    (900, 24, 20, 128, 24, True),
    (257, 33, 17, 256, 255, True),
    (1200, 40, 24, 256, 12, False),
    (300, 648, 520, 64, 20, False),  # 5265 tiles: one warp per whole tile
])
def test_tails_match_oracle(n, width, height, chunk, tail, ray):
    sc = scenes.random_scene(n=n, width=width, height=height, f=max(0.8 * max(width, height), 4.0), seed=n,
                             scale_range=(0.1, 0.6))
    sc.opacity = np.clip(sc.opacity * 0.3, 0.01, 0.99).astype(np.float32)
    cfg = RasterConfig(bg=(0.2, 0.1, 0.3), depth_ray=ray, chunk=chunk, fwd_tail=tail)
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
