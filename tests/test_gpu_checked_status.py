"""The checked build on lists that are corrupted all over: every CTA of every
kernel meets a failed index check, many of them while others are still
starting.  The kernels report it and end, what follows on the failed state
ends too, and the next forward is clean."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import numpy as np
import torch
sys.path.insert(0, {root!r})
from paper_2604_03092_gb300 import _abi, scenes
from paper_2604_03092_gb300.rasterizer import RasterConfig, Rasterizer

width, height, views, tile_w, tile_h, tail = {case}
sc = scenes.random_scene(n=6000, width=width, height=height, f=100.0 * width / 128, seed=3, n_views=views)
params = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (sc.means, sc.scales, sc.quats, sc.opacity, sc.rgb)]
rast = Rasterizer(sc.views, sc.n, RasterConfig(tile_w=tile_w, tile_h=tile_h, fwd_tail=tail))
clean = rast.forward(*params)
g = [torch.ones(3 * rast.n_pixels, device="cuda"), torch.ones(rast.n_pixels, device="cuda"), None, None]
for _ in range(20):
    rast.preprocess(*params)
    rast.bin_sort()
    n = int(rast.stats()["n_instances"])
    assert rast.status() == _abi.OK
    rast.ws_tensor(rast.layout.vals, n, torch.int32).fill_(-16)
    rast.render_fwd(rast.new_images())
    assert rast.status() == _abi.ERR_BOUNDS
    grads = rast.backward(*params, g)
    err = rast.max_error(torch.ones(rast.n_pixels, device="cuda"))
    assert rast.status() == _abi.ERR_BOUNDS
    assert all(float(t.abs().max()) == 0.0 for t in (*grads, err))
again = rast.forward(*params)
assert all(torch.equal(a, b) for a, b in zip(clean, again))
print("done")
"""


# half tiles on a full grid, and on few CTAs; whole tiles; every tile handed to the tail's kernel; 256-pixel tiles
@pytest.mark.parametrize("case", [(440, 330, 1, 8, 8, 0), (96, 72, 2, 8, 8, 0), (648, 520, 1, 8, 8, 0),
                                  (440, 330, 1, 8, 8, 255), (440, 330, 1, 16, 16, 0)])
def test_lists_corrupted_all_over(case):
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, case=case)], capture_output=True, text=True,
                       env=dict(os.environ, SPLAT2D_CHECKS="1"), timeout=1200)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
