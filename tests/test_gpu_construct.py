"""GPU parity of the tree-construction kernels (Algorithms 1 and 2) with the oracle.  Structure, tokens
and row ids must match exactly, values to fp32 rounding (they are stored as fp32).  The kernels take
their decisions (order of slot values, CDF search, v against t) in fp64 like the oracle, so a request
would be excused only where the oracle reports a decision within 1e-12 of its threshold."""
import numpy as np
import pytest

from oracle import dyspec_oracle as orc
from paper_2410_11744_b200 import workloads as wl

pytestmark = pytest.mark.gpu
EPS = {"order": 1e-12, "sample": 1e-12, "threshold": 1e-12}     # the kernels carry these sums and values in fp64


@pytest.fixture(scope="module")
def B():
    import torch
    assert torch.cuda.is_available()
    from paper_2410_11744_b200 import build
    build.build()
    from paper_2410_11744_b200 import binding
    return binding


def run_gpu(B, rows, uni, roots, m=None, threshold=None, max_nodes=None):
    import torch
    dev = "cuda:0"
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    n_req = len(roots)
    S = (m if threshold is None else max_nodes) + 1
    parents = torch.full((n_req, S), -9, dtype=torch.int32, device=dev)
    tokens = torch.full((n_req, S), -9, dtype=torch.int32, device=dev)
    nrows = torch.full((n_req, S), -9, dtype=torch.int32, device=dev)
    values = torch.zeros((n_req, S), dtype=torch.float32, device=dev)
    cvalues = torch.zeros((n_req, S), dtype=torch.float32, device=dev)
    n_nodes = torch.zeros((n_req,), dtype=torch.int32, device=dev)
    args = (t(rows), rows.shape[0], rows.shape[1], t(uni), len(uni), t(np.asarray(roots, np.int32)), n_req)
    if threshold is None:
        B.dyspec_build_tree_greedy(*args, m, parents, tokens, values, cvalues, nrows, n_nodes)
    else:
        B.dyspec_build_tree_threshold(*args, threshold, max_nodes, parents, tokens, values, cvalues, nrows, n_nodes)
    torch.cuda.synchronize()
    return [x.cpu().numpy() for x in (parents, tokens, values, cvalues, nrows, n_nodes)]


def compare(got, r, ref):
    parents, tokens, values, cvalues, nrows, n_nodes = got
    n = len(ref["parents"])
    assert int(n_nodes[r]) == n
    assert np.array_equal(parents[r, :n], ref["parents"])
    assert np.array_equal(tokens[r, :n], ref["tokens"])
    assert np.array_equal(nrows[r, :n], ref["rows"])
    assert np.allclose(values[r, :n], ref["values"], rtol=2e-5, atol=0)
    assert np.allclose(cvalues[r, :n], ref["child_values"], rtol=2e-5, atol=1e-30)


def excused(ref):
    return any(mg < EPS[kind] for kind, mg in ref["margins"])


@pytest.mark.parametrize("vocab,n_rows,m,sharp", [(32000, 24, 64, 3.0), (32768, 8, 40, 2.0), (1000, 64, 200, 2.0), (64, 16, 60, 1.0)])
def test_greedy_tree_matches_oracle(B, vocab, n_rows, m, sharp):
    rows, uni = wl.make_draft_table(100 + vocab, n_rows, vocab, sharp)
    roots = [0, 3, 5, 7]
    got = run_gpu(B, rows, uni, roots, m=m)
    skipped = 0
    for r, root in enumerate(roots):
        ref = orc.build_tree_greedy(rows, uni, m, root_row=root)
        if excused(ref):
            skipped += 1
            continue
        compare(got, r, ref)
    assert skipped == 0


@pytest.mark.parametrize("vocab,n_rows,threshold,cap,sharp", [(32000, 24, 0.02, 300, 3.0), (1000, 64, 0.004, 600, 2.0),
                                                              (64, 16, 0.01, 50, 1.0), (32000, 8, 0.5, 10, 3.0)])
def test_threshold_tree_matches_oracle(B, vocab, n_rows, threshold, cap, sharp):
    rows, uni = wl.make_draft_table(200 + vocab, n_rows, vocab, sharp)
    roots = [1, 2, 6]
    got = run_gpu(B, rows, uni, roots, threshold=threshold, max_nodes=cap)
    skipped = 0
    for r, root in enumerate(roots):
        ref = orc.build_tree_threshold(rows, uni, threshold, cap, root_row=root)
        if excused(ref):
            skipped += 1
            continue
        compare(got, r, ref)
    assert skipped == 0


def test_zipf_rows_give_deep_trees_and_match_oracle(B):
    rows, uni = wl.make_draft_table(77, 48, 32000, zipf=True)
    m = 96
    roots = list(range(8))
    got = run_gpu(B, rows, uni, roots, m=m)
    deepest = 0
    for r, root in enumerate(roots):
        ref = orc.build_tree_greedy(rows, uni, m, root_row=root)
        assert not excused(ref)
        compare(got, r, ref)
        depth = np.zeros(m + 1, int)
        for k in range(1, m + 1):
            depth[k] = depth[ref["parents"][k]] + 1
        deepest = max(deepest, int(depth.max()))
    assert deepest >= 3            # peaked rows give chains, flat rows give stars: both shapes are exercised


def _flat_and_peaked(seed, n_rows, vocab):
    """Every third row flat (its node becomes the centre of a star: one stream of hundreds of draws), the others peaked."""
    rows, uni = wl.make_draft_table(seed, n_rows, vocab, zipf=True)
    rng = np.random.default_rng(seed + 1)
    for i in range(0, n_rows, 3):
        p = rng.random(vocab) + 0.05
        rows[i] = (p / p.sum()).astype(np.float32)
    return rows, uni


# one and several row sums per lane (vocabularies at the edges 8192, 16384, 32768, and tiny ones), more requests than clusters
# of 8, 4 and 2 hold at once, more rows than a worker's tables were cut for, trees of one node and of the largest size
@pytest.mark.parametrize("vocab,n_rows,m,n_req", [(4, 3, 9, 2), (8192, 7, 70, 1), (8196, 7, 70, 1), (16384, 7, 70, 2), (16388, 7, 70, 2),
                                                  (32768, 5, 60, 1), (2000, 40, 33, 19), (2000, 40, 33, 40), (1000, 9, 20, 80),
                                                  (1000, 1, 40, 1), (512, 3000, 2047, 1), (4096, 900, 1, 1), (8192, 300, 1100, 1)])
def test_greedy_tree_at_the_edges_of_the_kernel(B, vocab, n_rows, m, n_req):
    rows, uni = _flat_and_peaked(vocab + m, n_rows, vocab)
    roots = [(5 * r) % n_rows for r in range(n_req)]
    got = run_gpu(B, rows, uni, roots, m=m)
    for r in sorted({0, n_req // 2, n_req - 1}):
        ref = orc.build_tree_greedy(rows, uni, m, root_row=roots[r])
        if not excused(ref):
            compare(got, r, ref)
        else:
            assert vocab == 4                                        # (so few tokens that equal slot values occur)


# short trees of more requests than run at once; trees with too many rows for the cluster that the requests leave them (the next with a
# hot CTA, or one CTA each): at each of the kernel's three row formats
@pytest.mark.parametrize("vocab,n_rows,m,n_req", [(4096, 40, 6, 18), (4096, 40, 24, 37), (9000, 40, 33, 74), (20000, 700, 400, 75),
                                                  (8192, 800, 700, 38), (9000, 800, 730, 24), (20000, 800, 700, 20), (2048, 2500, 2000, 106),
                                                  (9000, 2100, 2047, 31), (17000, 1900, 1850, 31), (17000, 1700, 1700, 19)])
@pytest.mark.parametrize("greedy", [True, False])
def test_trees_in_every_form(B, vocab, n_rows, m, n_req, greedy):
    rng = np.random.default_rng(vocab + m)
    rows = rng.random((n_rows, vocab), dtype=np.float32) ** 8                    # uneven enough for depth, and hundreds of children
    rows /= rows.sum(axis=1, keepdims=True)
    uni = rng.random(4099, dtype=np.float32)
    roots = [(5 * r) % n_rows for r in range(n_req)]
    threshold = 1e-7
    got = run_gpu(B, rows, uni, roots, m=m) if greedy else run_gpu(B, rows, uni, roots, threshold=threshold, max_nodes=m)
    for r in (0, n_req - 1):
        ref = orc.build_tree_greedy(rows, uni, m, root_row=roots[r]) if greedy else orc.build_tree_threshold(rows, uni, threshold, m, root_row=roots[r])
        assert not excused(ref)
        compare(got, r, ref)


@pytest.mark.parametrize("vocab,n_req,cap", [(2048, 1, 600), (9000, 20, 200), (20000, 1, 2047)])
def test_threshold_stream_through_a_collapsing_residual(B, vocab, n_req, cap):
    """Sixty tokens of probability 2^-1, 2^-2, ... and a tail of 1e-21: after some fifty draws what is left of the row is far
    below the rounding of any sum over the whole of it, and the draws that follow must still be the oracle's.  (Halving
    keeps 1 - r away from 0: a value v (1 - r) is only good to 1e-16 / (1 - r) in any fp64 implementation.)"""
    rng = np.random.default_rng(vocab)
    p = rng.random((2, vocab)) * 1e-24
    for i in range(2):
        p[i, rng.permutation(vocab)[:60]] = 0.5 ** np.arange(1, 61)
    rows, uni = p.astype(np.float32), rng.random(4099, dtype=np.float32)
    got = run_gpu(B, rows, uni, [r & 1 for r in range(n_req)], threshold=1e-25, max_nodes=cap)
    for r in (0, n_req - 1):
        ref = orc.build_tree_threshold(rows, uni, 1e-25, cap, root_row=r & 1)
        assert not excused(ref) and (ref["parents"] == 0).sum() > 100 and ref["values"][100] < 2.0 ** -50
        compare(got, r, ref)


def test_gpu_threshold_at_last_greedy_value_builds_the_same_tree(B):
    """The paper's statement (App. B), on the GPU alone: same set of root-to-node token paths."""
    rows, uni = wl.make_draft_table(9, 32, 4096, 3.0)
    m = 80
    g = run_gpu(B, rows, uni, [4], m=m)
    t = float(g[2][0, m])
    h = run_gpu(B, rows, uni, [4], threshold=t, max_nodes=4 * m)

    def paths(parents, tokens, n):
        out = set()
        for k in range(1, n):
            p, j = [], k
            while j > 0:
                p.append(int(tokens[j]))
                j = int(parents[j])
            out.add(tuple(reversed(p)))
        return out
    assert paths(g[0][0], g[1][0], int(g[5][0])) == paths(h[0][0], h[1][0], int(h[5][0]))


def test_constructed_tree_feeds_the_mask_builder(B):
    """The greedy tree's parent array is a legal input of the attention path (parents[i] < i)."""
    import torch
    rows, uni = wl.make_draft_table(3, 16, 2048, 2.5)
    m = 255
    got = run_gpu(B, rows, uni, [0], m=m)
    parents = np.ascontiguousarray(got[0][0])
    n = m + 1
    W = B.dyspec_words_per_row(n)
    bits = torch.zeros((n, W), dtype=torch.int32, device="cuda:0")
    depths = torch.zeros((n,), dtype=torch.int32, device="cuda:0")
    status = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    B.dyspec_build_tree_mask(torch.from_numpy(parents).to("cuda:0"), n, bits, depths, W, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref_bits, ref_depths = orc.build_tree_mask(parents, W)
    assert np.array_equal(bits.cpu().numpy().view(np.uint32), ref_bits)
    assert np.array_equal(depths.cpu().numpy(), ref_depths)


@pytest.mark.parametrize("greedy", [True, False])
@pytest.mark.parametrize("n_req", [1, 40, 150])
def test_a_wait_that_runs_out_is_reported(B, greedy, n_req):
    """With a bound of a nanosecond the wait for the first draw, whose row has yet to come from memory, cannot succeed: every request
    reports 0 nodes and the status word says why; the next call, with the usual bound, is right."""
    import torch
    vocab, n_rows, m = 32000, 16, 24
    rows, uni = wl.make_draft_table(11, n_rows, vocab, 3.0)
    roots = [r % n_rows for r in range(n_req)]
    dev = "cuda:0"
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    ints = [torch.full((n_req, m + 1), -9, dtype=torch.int32, device=dev) for _ in range(3)]
    vals = [torch.zeros((n_req, m + 1), device=dev) for _ in range(2)]
    n_nodes, status = torch.full((n_req,), -9, dtype=torch.int32, device=dev), torch.zeros(1, dtype=torch.int32, device=dev)
    head = (t(rows), n_rows, vocab, t(uni), len(uni), t(np.asarray(roots, np.int32)), n_req)
    tail = (ints[0], ints[1], vals[0], vals[1], ints[2], n_nodes)
    call = (lambda **k: B.dyspec_build_tree_greedy_bounded(*head, m, *tail, **k)) if greedy else \
           (lambda **k: B.dyspec_build_tree_threshold_bounded(*head, 1e-3, m, *tail, **k))
    call(wait_limit_ns=1, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == -6 and int(n_nodes.abs().max()) == 0
    status.zero_()
    call(status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = [x.cpu().numpy() for x in (ints[0], ints[1], vals[0], vals[1], ints[2], n_nodes)]
    for r in {0, n_req - 1}:
        ref = orc.build_tree_greedy(rows, uni, m, root_row=roots[r]) if greedy else orc.build_tree_threshold(rows, uni, 1e-3, m, root_row=roots[r])
        compare(got, r, ref)
    with pytest.raises(B.DyspecError):
        call(wait_limit_ns=-1)


@pytest.mark.parametrize("what", ["nan last", "nan inside", "inf inside", "no mass"])
@pytest.mark.parametrize("greedy", [True, False])
def test_rows_that_are_no_distributions_whatever_the_cluster(B, what, greedy):
    """Where a sum is no number the last token is drawn, with r = 0, and leaves the row; if it was the cause, the draws after it are
    ordinary ones again.  The same in hot CTAs, in clusters without one and in a single CTA."""
    rng = np.random.default_rng(3)
    vocab, m = 1000, 60
    rows = rng.random((12, vocab), dtype=np.float32) ** 4
    rows /= rows.sum(axis=1, keepdims=True)
    if what == "no mass":
        rows[::2] = 0.0
    else:
        rows[::2, vocab - 1 if what == "nan last" else vocab // 2] = np.inf if what == "inf inside" else np.nan
    uni = rng.random(4099, dtype=np.float32)
    trees = []
    for n_req in (1, 20, 40, 80):
        got = run_gpu(B, rows, uni, [0] * n_req, m=m) if greedy else run_gpu(B, rows, uni, [0] * n_req, threshold=1e-6, max_nodes=m)
        assert int(got[5].min()) == int(got[5].max()) == m + 1
        trees.append([x[n_req - 1] for x in got[:5]])
    assert trees[0][1][1] == vocab - 1
    if what == "nan last":
        assert len(set(trees[0][1][1:].tolist())) >= 4
    for t in trees[1:]:
        assert all(np.array_equal(t[i], trees[0][i]) for i in (0, 1, 4))
        assert np.allclose(t[2], trees[0][2], rtol=1e-6, atol=0) and np.allclose(t[3], trees[0][3], rtol=1e-6, atol=0)
