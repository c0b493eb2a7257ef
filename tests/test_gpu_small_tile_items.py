"""Small-tile kernel, many short items one after the other in the same CTA: items of one, two, an odd number of and more key
tiles than its shared-memory ring holds, so that an item begins at every place of the ring, a warp set has no tile at all, and
an item's epilogue meets its successor's first tiles.  Contiguous cache, and tree rows inside the pages at prefixes that
are no multiple of the tile (mask windows shifted).  Against the oracle; repeated on the same buffers, bit for bit."""
import numpy as np
import pytest

from oracle import dyspec_oracle as orc
from paper_2410_11744_b200 import workloads as wl

pytestmark = pytest.mark.gpu

MAX_ABS, MEAN_ABS = 2e-2, 2e-3       # as in test_gpu_parity.py
DEEPEST_RING = 8                     # stages, D = 64 (6 with D = 128)
# prefix, nodes (one query head per kv head): 1, 1, 2, 2, 1, 3, 9, 1, 2, 6, 16, 1 tiles of 64 keys
SHAPES = [(0, 1), (0, 64), (60, 4), (64, 64), (0, 3), (127, 40), (500, 64), (0, 64), (1, 64), (300, 33), (900, 17), (0, 2)]


@pytest.mark.parametrize("in_pages", [False, True])
@pytest.mark.parametrize("ctas, combine", [(1, 2 + 16), (3, 2 + 32), (3, 2 + 16), (7, 0)])
@pytest.mark.parametrize("d", [64, 128])
def test_many_short_items_in_a_cta(d, ctas, combine, in_pages):
    from paper_2410_11744_b200 import binding as B, build, runner as R
    build.build()
    rng = np.random.default_rng(d + ctas)
    w = wl.make_custom(45, 4, 4, d, [L for L, _ in SHAPES], [wl.random_tree(rng, n) for _, n in SHAPES])
    pw = wl.to_paged(w, 128, 3, tree_in_pages=True) if in_pages else None
    B.dyspec_set_tuning(0, ctas, combine)
    try:
        items, cta, info = B.dyspec_schedule_dry_run(4, 4, d, w.prefix_len, w.n_nodes, B.dyspec_words_per_row(64))
        batch = R.DeviceBatch(w, paged=pw)
    finally:
        B.dyspec_set_tuning(-1, 0, 2)
    tiles = [(items[cta[c]:cta[c + 1], 4] - items[cta[c]:cta[c + 1], 3]).tolist() for c in range(info["ctas"])]
    assert info["ctas"] == ctas == batch.plan.describe()["ctas"]
    assert {1, 2, 3, 9 if ctas < 7 else 6} <= set(sum(tiles, [])) and max(max(t) for t in tiles) > DEEPEST_RING
    assert any(t.count(1) >= 4 and t.count(2) >= 2 for t in tiles)
    if in_pages:
        ref = orc.tree_attention_paged(w.q, pw.k, pw.v, pw.page_table, 128, w.prefix_len, w.n_nodes, None, w.parents)
    else:
        ref = orc.tree_attention_ragged(w.q, w.k, w.v, w.prefix_len, w.n_nodes, w.kv_row_offset, w.parents)
    outs = []
    for _ in range(6):
        batch.out.zero_()
        batch.step()
        _, _, out_bits, status = batch.results()
        outs.append(out_bits)
        got = orc.bf16_bits_to_f64(out_bits)
        err = np.abs(got - ref)
        assert status == 0 and np.isfinite(got).all() and err.max() <= MAX_ABS and err.mean() <= MEAN_ABS, (err.max(), err.mean())
    assert all(np.array_equal(o, outs[0]) for o in outs[1:])
