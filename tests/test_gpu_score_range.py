"""Scores of every size that finite inputs give, up to near the end of fp32's range: where the softmax's exponent is formed
from a product and a reference that are both far larger than their difference.  Every score is exact in fp32 (rows of K are
one sign pattern times distinct bf16 numbers) and neighbours are at least 1 / 512 apart, so the oracle has one right answer."""
import numpy as np
import pytest

from oracle import dyspec_oracle as orc
from paper_2410_11744_b200 import workloads as wl

pytestmark = pytest.mark.gpu

MAX_ABS, MEAN_ABS = 2e-2, 2e-3       # as in test_gpu_parity.py


def _bits(x):
    u = np.ascontiguousarray(x, dtype=np.float32).view(np.uint32)
    assert not (u & 0xFFFF).any()    # the values are bf16 as they are
    return (u >> 16).astype(np.uint16)


@pytest.mark.parametrize("regime", [0, 1])
@pytest.mark.parametrize("ctas, combine", [(0, 2), (3, 0)])
@pytest.mark.parametrize("hq, hkv, d, n, L", [(4, 4, 64, 16, 128), (32, 32, 128, 64, 440), (8, 1, 128, 8, 300), (8, 8, 64, 33, 0)])
def test_scores_far_from_zero(hq, hkv, d, n, L, ctas, combine, regime):
    from paper_2410_11744_b200 import binding as B, build, runner as R
    build.build()
    rng = np.random.default_rng(n + d)
    w = wl.make_custom(61, hq, hkv, d, [L], [wl.greedy_tree(rng, n, 6, 0.3)])
    sign = np.where(rng.random(d) < 0.5, -1.0, 1.0)
    steps = np.concatenate([(1 + np.arange(128) / 128) * 2.0 ** e for e in range(4)])     # 512 distinct bf16 numbers
    side = np.where(rng.random((n, hq, 1)) < 0.5, -1.0, 1.0)      # rows whose largest score is the smallest in size, and negative
    for log2_score in (8, 20, 24, 27, 30, 31, 33, 40, 64, 110):   # of the smallest score, scale and log2(e) included
        for growing in (False, True):
            a = steps[:L + n] if growing else rng.permutation(steps)[:L + n]
            w.k[...] = _bits(sign * a[:, None, None] * np.ones((1, hkv, 1)))
            w.q[...] = _bits(sign * side * 2.0 ** (log2_score - round(np.log2(d) / 2 + 0.5)))
            ref = orc.tree_attention_ragged(w.q, w.k, w.v, w.prefix_len, w.n_nodes, w.kv_row_offset, w.parents)
            B.dyspec_set_tuning(regime, ctas, combine)
            try:
                batch = R.DeviceBatch(w)
            finally:
                B.dyspec_set_tuning(-1, 0, 2)
            batch.step()
            _, _, out_bits, status = batch.results()
            got = orc.bf16_bits_to_f64(out_bits)
            assert status == 0 and np.isfinite(got).all(), (log2_score, growing)
            err = np.abs(got - ref)
            assert err.max() <= MAX_ABS and err.mean() <= MEAN_ABS, (log2_score, growing, err.max(), err.mean())
