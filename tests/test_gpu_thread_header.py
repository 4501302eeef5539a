"""Reading the status from a thread keeps a page-locked block for that thread.
Giving it back when the thread ends does not disturb a graph that another
thread is capturing."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import threading
import numpy as np
import torch
sys.path.insert(0, {root!r})
from paper_2604_03092_gb300 import _abi, scenes
from paper_2604_03092_gb300.rasterizer import Rasterizer

def problem(seed):
    sc = scenes.random_scene(n=2000, width=96, height=72, f=70.0, seed=seed)
    params = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (sc.means, sc.scales, sc.quats, sc.opacity, sc.rgb)]
    rast = Rasterizer(sc.views, sc.n)
    return rast, params, rast.forward(*params)

rast, params, want = problem(3)
other, other_params, _ = problem(4)
out = rast.new_images()
torch.cuda.synchronize()
capturing, read = threading.Event(), threading.Event()
status = []

def reader():
    with torch.cuda.stream(torch.cuda.Stream()):
        status.append(other.status())
        read.set()
        capturing.wait(60)

t = threading.Thread(target=reader)
t.start()
assert read.wait(60)
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    rast.forward(*params, out=out, check=False)
    capturing.set()
    t.join()
    rast.forward(*params, out=out, check=False)
graph.replay()
torch.cuda.synchronize()
assert status == [_abi.OK] and rast.status() == _abi.OK
assert all(torch.equal(a, b) for a, b in zip(out, want))
print("done")
"""


def test_a_reading_thread_ends_during_a_capture():
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
