"""The one-warp sort of short tile buckets: lengths around its rounds of 32
and its limit of 256, one radix pass and two, tie runs ranked as they are
written out and runs too long for that, bit-exact against the oracle."""
import numpy as np
import pytest

from paper_2604_03092_gb300 import scenes
from test_gpu_parity import _check_bin_sort

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 255, 256, 257])
@pytest.mark.parametrize("depths", ["spread", "one", "few", "near"])
def test_one_tile_bucket(n, depths):
    # every surfel lies before the 8x8 image, so its one tile holds n entries
    sc = scenes.random_scene(n=n, width=8, height=8, f=8.0, seed=n, xy_range=0.2, scale_range=(0.05, 0.1), n_views=1,
                             with_target=False)
    rng = np.random.default_rng(n)
    z = {"spread": rng.uniform(2.0, 4.0, n),                        # 23 varying bits: two passes
         "one": np.full(n, 3.0),                                    # no varying bit: one run of n
         "few": np.float32(3.0) + rng.integers(0, 40, n) * 2e-7,    # a few ulps: one pass, runs of several
         "near": np.where(np.arange(n) % 3 == 0, 2.0, 3.0 + rng.uniform(0, 1e-4, n))}[depths]
    sc.means[:, 2] = z.astype(np.float32)
    sc.opacity[:] = 0.9
    counts = _check_bin_sort(sc, (8, 8))
    assert counts.max() >= 0.9 * n - 1


def test_many_short_buckets():
    # 3 views of 6,400 tiles: several sweeps of the scan, empty tiles among them
    sc = scenes.random_scene(n=6000, width=640, height=640, f=400.0, seed=3, n_views=3, with_target=False,
                             scale_range=(0.005, 0.05))
    counts = _check_bin_sort(sc, (8, 8))
    assert (counts == 0).any() and counts.max() < 256
