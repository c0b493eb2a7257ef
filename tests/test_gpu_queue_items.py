"""Items of the shared work queue that follow one another closely: of one key tile, with one query half and with two in
every order, with and without tile skipping, so that an item's epilogue, its successor's first scores and its last
product meet in all ways.  Compared with the oracle; run twice on the same buffers."""
import numpy as np
import pytest

from oracle import dyspec_oracle as orc
from paper_2410_11744_b200 import workloads as wl

pytestmark = pytest.mark.gpu

MAX_ABS, MEAN_ABS = 2e-2, 2e-3       # as in test_gpu_parity.py


@pytest.mark.parametrize("d, sparse", [(128, False), (128, True), (64, False)])
def test_short_items_of_one_and_two_halves(d, sparse):
    from paper_2410_11744_b200 import binding as B, build, runner as R
    build.build()
    rng = np.random.default_rng(d)
    shapes = [(0, 1), (0, 128), (1, 129), (127, 65), (128, 257), (0, 256), (300, 100), (129, 700)]   # prefix, nodes (one head per kv head)
    trees = [wl.random_tree(rng, n) for _, n in shapes]
    w = wl.make_custom(41, 24, 24, d, [L for L, _ in shapes], trees)
    B.dyspec_set_tuning(1, 0, 2)
    try:
        batch = R.DeviceBatch(w, sparse=sparse)
    finally:
        B.dyspec_set_tuning(-1, 0, 2)
    info = batch.plan.describe()
    assert info["dynamic"] == 1 and info["groups"] > info["ctas"]
    ref = orc.tree_attention_ragged(w.q, w.k, w.v, w.prefix_len, w.n_nodes, w.kv_row_offset, w.parents)
    for _ in range(2):
        batch.out.zero_()
        batch.step()
        _, _, out_bits, status = batch.results()
        got = orc.bf16_bits_to_f64(out_bits)
        err = np.abs(got - ref)
        assert status == 0 and np.isfinite(got).all() and err.max() <= MAX_ABS and err.mean() <= MEAN_ABS, (err.max(), err.mean())
