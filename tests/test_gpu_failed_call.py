"""A call whose launch the runtime refuses (here, on a stream whose capture
has become invalid) reports it, and leaves nothing behind: the calls after it
succeed."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes
import sys
import numpy as np
import torch
sys.path.insert(0, {root!r})
from paper_2604_03092_gb300 import _abi, scenes
from paper_2604_03092_gb300.rasterizer import RasterConfig, Rasterizer

lib = _abi.load()
sc = scenes.random_scene(n=500, width=64, height=48, f=50.0, seed=3)
params = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (sc.means, sc.scales, sc.quats, sc.opacity, sc.rgb)]
rast = Rasterizer(sc.views, sc.n, RasterConfig(tile_w=16, tile_h=16, chunk=64))
want = rast.forward(*params)
out, grads, err = rast.new_images(), rast.new_grads(), torch.rand(rast.n_pixels, device="cuda")
worst = torch.zeros(sc.n, device="cuda")
n = 1000
alpha, keep = torch.rand(n, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
count = torch.empty(1, dtype=torch.int64, device="cuda")
tmp = torch.empty(4096, dtype=torch.uint8, device="cuda")
row = torch.tensor([[1.0, 0, 0, 0, 0, 0, 0, 1]], device="cuda")
moved = [t.clone() for t in (params[0], params[2], params[1])]
keys = torch.arange(n, device="cuda").flip(0).contiguous()
ref = ctypes.byref
cfg, prob, sf = ref(rast._cfg), ref(rast._prob), ref(rast._sf)
ws, size = rast._ws_ptr, rast.ws_bytes
images = [t.data_ptr() for t in out]

calls = {{
    "forward": lambda s: lib.splat2d_forward(cfg, prob, sf, ws, size, *images, None, s),
    "gate": lambda s: lib.splat2d_accum_gate(alpha.data_ptr(), n, 0.5, keep.data_ptr(), count.data_ptr(), tmp.data_ptr(),
                                             tmp.numel(), s),
    "bin_sort": lambda s: lib.splat2d_bin_sort(cfg, prob, ws, size, s),
    "max_error": lambda s: lib.splat2d_max_error(cfg, prob, ws, size, err.data_ptr(), worst.data_ptr(), s),
    "sim3": lambda s: lib.splat2d_sim3_apply(sc.n, moved[0].data_ptr(), moved[1].data_ptr(), moved[2].data_ptr(),
                                             row.data_ptr(), None, s),
    "sort": lambda s: lib.splat2d_sort_pairs_noalloc(keys.data_ptr(), keep.data_ptr(), n, 16, s),
}}
good, bad = torch.cuda.Stream(), torch.cuda.Stream()
torch.cuda.synchronize()
for call in calls.values():  # what a first call looks up is there
    assert call(good.cuda_stream) == _abi.OK
torch.cuda.synchronize()
for name, call in calls.items():
    for after in ("forward", "sim3"):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(bad):
            graph.capture_begin()
            try:
                torch.cuda.synchronize()  # not allowed here: the capture is invalid from now on
            except RuntimeError:
                pass
            assert call(bad.cuda_stream) == _abi.ERR_CUDA, name
            try:
                graph.capture_end()
            except RuntimeError:
                pass
        assert calls[after](good.cuda_stream) == _abi.OK, (name, after)
torch.cuda.synchronize()
assert all(torch.equal(a, b) for a, b in zip(out, want))
print("done")
"""


def test_calls_after_a_refused_one_succeed():
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
