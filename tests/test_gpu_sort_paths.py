"""The radix sort's block shapes change with the size: 8-bit passes take
4096-pair tiles below 2,490,368 pairs and 8192-pair tiles from there on, 9-bit
passes 4096-pair tiles, so a 17-bit sort mixes both.  Sizes on both sides of
the change, with ragged tails, against numpy's stable argsort, exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SMALL = 2 * 152 * 8192


@pytest.mark.parametrize("n", [8191, 8193, SMALL - 1, SMALL, SMALL + 4097])
@pytest.mark.parametrize("bits", [8, 17, 18, 26])
def test_sort_across_block_shapes(n, bits):
    import torch
    from paper_2409_08270_gb300 import build, flashsplat
    build.build()
    rng = np.random.default_rng(n + bits)
    keys = rng.integers(0, 1 << bits, n, dtype=np.uint64).astype(np.uint32)
    keys[n // 3: n // 2] = keys[0]  # one digit fills whole tiles
    vals = rng.permutation(n).astype(np.uint32)
    order = np.argsort(keys, kind="stable")
    k = torch.from_numpy(keys.view(np.int32).copy()).cuda()
    v = torch.from_numpy(vals.view(np.int32).copy()).cuda()
    flashsplat.fs_test_sort_pairs(0, k, v, bits)
    np.testing.assert_array_equal(k.cpu().numpy().view(np.uint32), keys[order])
    np.testing.assert_array_equal(v.cpu().numpy().view(np.uint32), vals[order])
