"""Ordered compactions of the mapping kernels (accumulation gate, adaptive
voxelization) at the edges of their blocks' sums: one block, a last block with
one element, ragged columns and rows, and either side of the number of blocks
up to which each block adds up the counts before its own."""
import numpy as np
import pytest
import torch

import oracle
from oracle import fusion
from paper_2604_03092_gb300 import mapping
from paper_2604_03092_gb300.rasterizer import accum_gate
from test_gpu_mapping import _map

pytestmark = pytest.mark.gpu

GATE_TILE, VOX_TILE, SUM_BLOCKS = 1024, 256, 4096


@pytest.mark.parametrize("n", [255, 257, 1025, 2 * GATE_TILE, SUM_BLOCKS * GATE_TILE, SUM_BLOCKS * GATE_TILE + 1])
@pytest.mark.parametrize("tau", [0.0, 0.4, 2.0])  # none, some, all but NaN
def test_gate_across_blocks(n, tau):
    a = np.random.default_rng(n).uniform(0, 1, n).astype(np.float32)
    a[3::11] = np.float32("nan")
    keep, n_keep = accum_gate(torch.from_numpy(a).cuda(), tau)
    expect = oracle.accum_gate(a, np.float32(tau))
    assert int(n_keep) == expect.size
    np.testing.assert_array_equal(keep[:expect.size].cpu().numpy().astype(np.int64), expect)


@pytest.mark.parametrize("W,H", [(2, 2), (3, 1), (1, 5), (2 * VOX_TILE, 2), (2 * VOX_TILE + 1, 3), (33, 64)])
def test_voxelize_across_blocks(W, H):
    m, q, s, o, c = _map(W, H, W + 100 * H, 0.1)
    got, block, n_out = mapping.voxelize(*(torch.from_numpy(a).cuda() for a in (m, q, s, o, c)), W, H, 0.1)
    ref, ref_block = fusion.voxelize(m, q, s, o, c, W, H, 0.1)
    k = ref_block.size
    assert int(n_out) == k
    np.testing.assert_array_equal(block[:k].cpu().numpy(), ref_block)
    for g, r in zip(got, ref):
        np.testing.assert_allclose(g[:k].cpu().numpy().astype(np.float64).reshape(r.shape), r, rtol=2e-6, atol=1e-7)


@pytest.mark.parametrize("H", [2 * SUM_BLOCKS, 2 * SUM_BLOCKS + 1])
def test_voxelize_many_blocks(H):
    """Rows of 256 blocks, so as many counts as rows of blocks; every value an
    integer below 2^22, so the means of four are exact."""
    W, nb = 2 * VOX_TILE, VOX_TILE * ((H + 1) // 2)
    rng = torch.Generator(device="cuda").manual_seed(H)
    ints = lambda *shape: torch.randint(0, 1 << 20, shape, device="cuda", generator=rng).float()
    means, scales, opacity, rgb = ints(H * W, 3), ints(H * W, 2), ints(H * W), ints(H * W, 3)
    rows = torch.arange(H * W, device="cuda")
    at = (rows // W) // 2 * VOX_TILE + (rows % W) // 2
    split = torch.rand(nb, device="cuda", generator=rng) < 0.5
    means[:, 2] = torch.where(split[at], rows.float() % 97 * 4 + (rows // W % 2) * 400, 5.0)
    quats = torch.zeros(H * W, 4, device="cuda")
    quats[:, 0] = 1.0
    got, block, n_out = mapping.voxelize(means, quats, scales, opacity, rgb, W, H, 0.5)
    member = torch.argsort(at, stable=True)  # blocks in order, their primitives in row-major order
    kept = split[at[member]]
    first = torch.ones_like(kept)
    first[1:] = at[member][1:] != at[member][:-1]
    out = member[kept | first]
    k = out.numel()
    assert int(n_out) == k and torch.equal(block[:k].long(), at[out])
    size = torch.bincount(at, minlength=nb)
    for g, x in zip((got[0], got[2], got[3], got[4]), (means, scales, opacity, rgb)):
        x = x.reshape(H * W, -1)
        mean = torch.zeros(nb, x.shape[1], device="cuda", dtype=torch.float64).index_add_(0, at, x.double())
        mean = (mean / size[:, None]).float()
        want = torch.where(split[at[out]][:, None], x[out], mean[at[out]])
        assert torch.equal(g[:k].reshape(k, -1), want)
    assert torch.equal(got[1][:k], quats[:k])
