"""The single-request entry point keeps one workspace for every (prefix, tree) size of a shape.  Sizes whose split groups count
arrivals in that workspace, called in turn with sizes whose partials reach further into it, must each find their
counters at zero: every output equals the ragged entry point's, which has a workspace of its own."""
import numpy as np
import pytest

from paper_2410_11744_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def test_sizes_that_share_the_workspace_do_not_share_their_counters():
    import torch
    assert torch.cuda.is_available()
    from paper_2410_11744_b200 import build
    build.build()
    from paper_2410_11744_b200 import binding as B, runner as R
    hq, hkv, d = 64, 8, 128
    rng = np.random.default_rng(9)
    sizes = [(4200, 20), (4100, 90), (900, 48), (3500, 90), (4200, 20), (5000, 30), (4100, 90), (4200, 20)]
    W = B.dyspec_words_per_row(90)
    B.dyspec_release_cache()
    B.dyspec_set_default_shape(hq, hkv, d, W, 0.0)
    made, counted = {}, set()
    for L, n in sizes:
        if (L, n) not in made:
            b = R.DeviceBatch(wl.make_custom(L + n, hq, hkv, d, [L], [wl.greedy_tree(rng, n, 6, 0.3)]), words_per_row=W)
            b.step()
            made[(L, n)] = b
            if b.plan.describe()["split_groups"]:
                counted.add(b.plan.workspace_bytes())
    assert len(counted) >= 2                                  # otherwise nothing here counts arrivals at different places
    for L, n in sizes:
        b = made[(L, n)]
        out = torch.zeros_like(b.out)
        for _ in range(2):
            B.dyspec_tree_attention(b.q, b.k, b.v, L, b.bits, n, out)
        torch.cuda.synchronize()
        assert torch.equal(out, b.out), (L, n)
    B.dyspec_release_cache()
