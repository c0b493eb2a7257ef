"""The mask builder at the edges of its row blocks (32 rows a warp, 512 a CTA), with rows wider than the tree needs and with
requests of very different sizes in one batch: bits, depths and tile sets exactly as the oracle's."""
import numpy as np
import pytest

from oracle import dyspec_oracle as orc
from paper_2410_11744_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,W", [([1], 4), ([31, 32, 33], 4), ([127, 128, 129, 1], 8), ([511, 512, 513], 20), ([1023, 1024], 32), ([128], 64), ([0, 5, 0, 256, 257], 12),
                                     ([2047, 3, 2048, 640], 64)])
@pytest.mark.parametrize("shape", ["random", "chain", "star"])
def test_mask_rows_at_block_edges(sizes, W, shape):
    import torch
    from paper_2410_11744_b200 import build
    build.build()
    from paper_2410_11744_b200 import binding as B
    rng = np.random.default_rng(len(sizes) * 100 + W)
    make = {"random": lambda n: wl.random_tree(rng, n), "chain": lambda n: np.arange(-1, n - 1, dtype=np.int32),
            "star": lambda n: np.concatenate([[-1], np.zeros(n - 1, np.int32)]).astype(np.int32)}[shape]
    trees = [make(n) if n else np.zeros(0, np.int32) for n in sizes]
    total = sum(sizes)
    parents = torch.from_numpy(np.concatenate(trees).astype(np.int32)).to("cuda:0")
    rows = [10 + n for n in sizes]
    plan = B.Plan(4, 4, 64, [10] * len(sizes), sizes, np.concatenate([[0], np.cumsum(rows)[:-1]]).tolist(), sum(rows), W, 0.0)
    bits = torch.full((total, W), -1, dtype=torch.int32, device="cuda:0")
    depths, tiles = torch.full((total,), -1, dtype=torch.int32, device="cuda:0"), torch.full((total,), -1, dtype=torch.int32, device="cuda:0")
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    B.dyspec_plan_build_tree_mask_tiles(plan, parents, bits, depths, tiles, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got, at = bits.cpu().numpy().view(np.uint32), 0
    for tree in trees:
        n = len(tree)
        if n:
            ref_bits, ref_depths = orc.build_tree_mask(tree, W)
            assert np.array_equal(got[at:at + n], ref_bits)
            assert np.array_equal(depths.cpu().numpy()[at:at + n], ref_depths)
            ref_tiles = np.zeros(n, np.uint32)
            for t in range(W // 2):
                ref_tiles |= (ref_bits[:, 2 * t:2 * t + 2] != 0).any(axis=1).astype(np.uint32) << np.uint32(t)
            assert np.array_equal(tiles.cpu().numpy().view(np.uint32)[at:at + n], ref_tiles)
        at += n
