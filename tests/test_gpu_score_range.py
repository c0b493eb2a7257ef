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


@pytest.mark.parametrize("d", [64, 128])
def test_scores_at_the_end_of_the_range(d):
    """Small-tile kernel, a given scale above 1 / log2(e): scaled scores up to a tenth below 2^128, all of them finite."""
    import torch
    from paper_2410_11744_b200 import binding as B, build
    build.build()
    L, n, H, scale = 8, 5, 4, 40.0
    rng = np.random.default_rng(d)
    w = wl.make_custom(62, H, H, d, [L], [wl.greedy_tree(rng, n, 3, 0.3)])
    sign = np.where(rng.random(d) < 0.5, -1.0, 1.0)
    side = np.where(rng.random((n, H, 1)) < 0.5, -1.0, 1.0)
    a = 1 + rng.permutation(L + n) / 128
    w.k[...] = _bits(sign * a[:, None, None] * np.ones((1, H, 1)))
    w.q[...] = _bits(sign * side * 2.0 ** 122 / d)              # scores 2^122 * a, times 40 log2(e) = 2^127.85 * a
    assert 2.0 ** 122 * a.max() * scale * np.log2(np.e) < 2.0 ** 128
    ref = orc.tree_attention_ragged(w.q, w.k, w.v, w.prefix_len, w.n_nodes, w.kv_row_offset, w.parents, scale=scale)
    t = lambda x, kind=torch.bfloat16: torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0").view(kind)
    q, k, v = t(w.q.view(np.int16)), t(w.k.view(np.int16)), t(w.v.view(np.int16))
    W = B.dyspec_words_per_row(n)
    B.dyspec_set_tuning(0, 0, 2)
    try:
        plan = B.Plan(H, H, d, w.prefix_len, w.n_nodes, w.kv_row_offset, L + n, W, scale)
    finally:
        B.dyspec_set_tuning(-1, 0, 2)
    bits, depths, status = (torch.zeros(s, dtype=torch.int32, device="cuda:0") for s in ((n, W), (n,), (1,)))
    out = torch.zeros_like(q)
    workspace = torch.zeros(max(256, plan.workspace_bytes()), dtype=torch.uint8, device="cuda:0")
    B.dyspec_plan_build_tree_mask(plan, t(w.parents[0], torch.int32), bits, depths, status)
    B.dyspec_tree_attention_ragged(plan, q, k, v, bits, out, workspace, None, status)
    torch.cuda.synchronize()
    err = np.abs(out.float().cpu().numpy() - ref)
    assert int(status.item()) == 0 and err.max() <= MAX_ABS and err.mean() <= MEAN_ABS, (err.max(), err.mean())
