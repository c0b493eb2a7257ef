"""Items of the tensor-core kernel's shared work queue (longest first) that are short, so that an item's epilogue, its
successor's first scores and its last product lie close together, with one and with two query halves.  ONE_TILE: mostly
items of one key tile, about four a CTA behind a few longer ones, both kinds mixed.  FEW_TILES: one or two to eight key tiles,
two halves only from two tiles on.  With and without tile skipping; against the oracle, twice on the same buffers."""
from collections import Counter

import numpy as np
import pytest

from oracle import dyspec_oracle as orc
from paper_2410_11744_b200 import workloads as wl

pytestmark = pytest.mark.gpu

MAX_ABS, MEAN_ABS = 2e-2, 2e-3       # as in test_gpu_parity.py
# query heads, kv heads, (prefix, nodes) of the requests
FEW_TILES = (24, 24, [(0, 1), (0, 128), (1, 129), (127, 65), (128, 257), (0, 256), (300, 100), (129, 700)])
ONE_TILE = (192, 24, 3 * [(0, 1), (0, 16), (0, 17), (0, 32), (0, 32), (0, 33), (0, 24), (1, 20), (128, 16), (129, 32), (300, 10), (127, 64)])


def _item_mix(B, hq, hkv, d, shapes):
    """{(key tiles, query halves): items} of the schedule, and its CTAs."""
    ns = [n for _, n in shapes]
    items, _, info = B.dyspec_schedule_dry_run(hq, hkv, d, [L for L, _ in shapes], ns, B.dyspec_words_per_row(max(ns)))
    rows = lambda it: min(256, ns[it[0]] * (hq // hkv) - it[2])
    return Counter((int(it[4] - it[3]), 2 if rows(it) > 128 else 1) for it in items), info["ctas"]


@pytest.mark.parametrize("d, sparse", [(128, False), (128, True), (64, False)])
@pytest.mark.parametrize("kind", ["few_tiles", "one_tile"])
def test_short_items_of_one_and_two_halves(kind, d, sparse):
    from paper_2410_11744_b200 import binding as B, build, runner as R
    build.build()
    rng = np.random.default_rng(d)
    hq, hkv, shapes = FEW_TILES if kind == "few_tiles" else ONE_TILE
    trees = [wl.random_tree(rng, n) for _, n in shapes]
    w = wl.make_custom(41, hq, hkv, d, [L for L, _ in shapes], trees)
    B.dyspec_set_tuning(1, 0, 2)
    try:
        batch = R.DeviceBatch(w, sparse=sparse)
        mix, ctas = _item_mix(B, hq, hkv, d, shapes)
    finally:
        B.dyspec_set_tuning(-1, 0, 2)
    info = batch.plan.describe()
    assert info["dynamic"] == 1 and info["groups"] > info["ctas"] == ctas and sum(mix.values()) == info["groups"]
    if kind == "few_tiles":
        assert {(1, 1), (2, 1), (2, 2), (3, 2), (4, 1), (4, 2), (6, 2), (8, 2)} <= set(mix)
    else:
        assert {(1, 1), (1, 2), (2, 1), (2, 2), (3, 2), (4, 1)} == set(mix)
        assert mix[1, 1] > ctas and mix[1, 2] > 2 * ctas
    ref = orc.tree_attention_ragged(w.q, w.k, w.v, w.prefix_len, w.n_nodes, w.kv_row_offset, w.parents)
    for _ in range(2):
        batch.out.zero_()
        batch.step()
        _, _, out_bits, status = batch.results()
        got = orc.bf16_bits_to_f64(out_bits)
        err = np.abs(got - ref)
        assert status == 0 and np.isfinite(got).all() and err.max() <= MAX_ABS and err.mean() <= MEAN_ABS, (err.max(), err.mean())
