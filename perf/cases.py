"""Workloads whose speed matters to a user of the library, and how each is set up and run.

A serving step of speculative decoding grows a draft tree, builds its mask, runs tree attention in every layer,
verifies the tree and keeps the accepted rows.  The cases below are those parts, alone and together, through the
public entry points (`paper_2410_11744_b200.binding`), from one tiny request to a ragged batch, with the shapes of
the repository's benchmark and tests.  `op` says which part a case is:

  attend   mask build, then `layers` tree-attention calls, each layer with its own Q, K, V and output.  The plan is
           kept: all layers and steps of one batch structure share it.  layout: contiguous, paged (tree rows
           outside the pages) or in_pages (tree rows appended to the paged sequence).  dfs: the token order is
           renumbered first and the attention skips empty tree tiles.
  loop     a single-request decoding loop through the convenience entry point: the prefix grows and the tree
           changes at every step, so each step brings the library a shape that it has not planned yet.
  verify   Algorithm 3 over a batch of trees with the draft and target rows of every node.
  grow     Algorithm 1 (greedy) or 2 (threshold) over a table of draft distributions.
  decode   one whole step of a batch with a paged cache: grow, plan, mask, attention, verify, compaction.  The plan
           and its workspace are made inside: the batch structure is new at every step.

Sizes of ragged batches come from the case (`shape_seed`), so that its work is known; everything else comes from
the seed that `prepare` is given.
"""
import heapq
import math
import random

import numpy as np
import torch

from paper_2410_11744_b200 import binding as B
from paper_2410_11744_b200 import workloads

DEV = "cuda"


def listed():
    return [
        # the smallest request of the test suite: nothing but launches and latency
        dict(name="tiny_request", op="attend", hq=4, hkv=4, d=64, n_req=1, l_lo=128, l_hi=128, n_lo=16, n_hi=16,
             layers=1, layout="contiguous", dfs=False, page=0, alpha=0.3, shape_seed=0),
        # one chat request with the paper's usual 64-node tree, MHA; eight layers of a model
        dict(name="chat_mha_64", op="attend", hq=32, hkv=32, d=128, n_req=1, l_lo=1024, l_hi=1024, n_lo=64, n_hi=64,
             layers=8, layout="contiguous", dfs=False, page=0, alpha=0.3, shape_seed=0),
        # a serving batch of small trees at odd prefix lengths, tree rows appended to the pages: streams K and V
        dict(name="serve_small_trees", op="attend", hq=32, hkv=32, d=128, n_req=16, l_lo=200, l_hi=4096, n_lo=16,
             n_hi=64, layers=2, layout="in_pages", dfs=False, page=256, alpha=0.3, shape_seed=5),
        # long context and a large, deep tree, MHA: bytes and operations weigh about the same
        dict(name="long_mha_256", op="attend", hq=32, hkv=32, d=128, n_req=1, l_lo=4096, l_hi=4096, n_lo=256,
             n_hi=256, layers=4, layout="contiguous", dfs=False, page=0, alpha=0.1, shape_seed=0),
        # one request with a large tree, GQA 8, paged cache: dense contraction
        dict(name="gqa_512_paged", op="attend", hq=64, hkv=8, d=128, n_req=1, l_lo=2048, l_hi=2048, n_lo=512,
             n_hi=512, layers=4, layout="paged", dfs=False, page=256, alpha=0.3, shape_seed=0),
        # the benchmark's default: ragged batch of 8, GQA 8, prefixes 512 - 8192, trees of 32 - 768 nodes
        dict(name="ragged8_gqa", op="attend", hq=64, hkv=8, d=128, n_req=8, l_lo=512, l_hi=8192, n_lo=32, n_hi=768,
             layers=2, layout="contiguous", dfs=False, page=0, alpha=0.3, shape_seed=5),
        # the paper's random-tree experiment at its largest size: renumber, mask with tile sets, skip empty tiles
        dict(name="random_tree_2048", op="attend", hq=64, hkv=64, d=128, n_req=1, l_lo=0, l_hi=0, n_lo=2048,
             n_hi=2048, layers=1, layout="contiguous", dfs=True, page=0, alpha=0.0, shape_seed=0),
        # single-request decoding loop: ten steps of a growing prefix, odd sizes, two layers each
        dict(name="single_loop", op="loop", hq=32, hkv=32, d=128, l_lo=715, n_lo=48, steps=10, layers=2, alpha=0.3),
        # verification of one 64-node tree, Llama2's vocabulary, a draft that is often right
        dict(name="verify_one", op="verify", n_req=1, n_lo=64, n_hi=64, vocab=32000, gap=0.3, bonus=True, shape_seed=0),
        # a batch of layer-wise trees bounded by a threshold
        dict(name="grow_threshold_8", op="grow", algo="threshold", n_req=8, m=512, vocab=32000, rows=256,
             threshold=0.002),
        # the paper's largest tree, built greedily for one request
        dict(name="grow_greedy_768", op="grow", algo="greedy", n_req=1, m=768, vocab=32000, rows=256, threshold=0.0),
        # a whole step of a batch of 8, GQA 8, four layers: every component once, the plan made on the way
        dict(name="decode_batch8", op="decode", hq=64, hkv=8, d=128, n_req=8, l_lo=512, l_hi=4096, m=127, layers=4,
             page=256, vocab=32000, rows=256, gap=0.3, shape_seed=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["attend"] * 6 + ["loop", "verify", "verify", "grow", "grow", "decode"])
    seed = rng.randrange(1 << 20)
    if op == "attend":
        hq, hkv, d = rng.choice([(32, 32, 128), (64, 8, 128), (32, 8, 128), (16, 8, 64), (8, 8, 64), (64, 64, 128)])
        n_req = _log_int(rng, 1, 16)
        n_hi = _log_int(rng, 8, min(768, 3000 // n_req) if hq > 16 else 512)
        l_hi = _log_int(rng, 100, 8192 if n_req * n_hi * hq <= 8 * 400 * 64 else 2048)
        layout = rng.choice(["contiguous", "contiguous", "paged", "in_pages"])
        dfs = n_req == 1 and layout == "contiguous" and rng.random() < 0.4
        if dfs:
            n_hi, l_hi = _log_int(rng, 256, 2048), rng.choice([0, _log_int(rng, 16, 1024)])
        return dict(op=op, hq=hq, hkv=hkv, d=d, n_req=n_req, l_lo=max(0, l_hi // rng.choice([1, 4, 16])), l_hi=l_hi,
                    n_lo=max(1, n_hi // rng.choice([1, 2, 8])), n_hi=n_hi, layers=rng.choice([1, 2, 4]), layout=layout,
                    dfs=dfs, page=0 if layout == "contiguous" else rng.choice([128, 256, 512]),
                    alpha=0.0 if dfs else rng.choice([0.1, 0.3, 1.0]), shape_seed=seed)
    if op == "loop":
        hq, hkv, d = rng.choice([(32, 32, 128), (64, 8, 128), (32, 8, 128), (16, 8, 64)])
        return dict(op=op, hq=hq, hkv=hkv, d=d, l_lo=_log_int(rng, 64, 4096), n_lo=_log_int(rng, 8, 256),
                    steps=rng.randint(3, 12), layers=rng.choice([1, 2, 4]), alpha=rng.choice([0.1, 0.3, 1.0]))
    vocab = rng.choice([32000, 32000, 8192, 1024, 4 * rng.randint(500, 8000)])
    if op == "verify":
        n_req = _log_int(rng, 1, 16)
        n_hi = _log_int(rng, 16, 256)
        return dict(op=op, n_req=n_req, n_lo=max(2, n_hi // 2), n_hi=n_hi, vocab=vocab,
                    gap=math.exp(rng.uniform(math.log(0.05), math.log(1.0))), bonus=rng.random() < 0.5, shape_seed=seed)
    if op == "grow":
        algo = rng.choice(["greedy", "threshold"])
        return dict(op=op, algo=algo, n_req=_log_int(rng, 1, 16), m=_log_int(rng, 16, 768 if algo == "greedy" else 1024),
                    vocab=vocab, rows=rng.choice([64, 256]), threshold=0.0 if algo == "greedy" else 10.0 ** rng.uniform(-3, -2))
    hq, hkv, d = rng.choice([(64, 8, 128), (32, 32, 128), (32, 8, 128)])
    return dict(op=op, hq=hq, hkv=hkv, d=d, n_req=_log_int(rng, 1, 8), l_lo=200, l_hi=_log_int(rng, 300, 4096),
                m=_log_int(rng, 16, 127), layers=rng.choice([2, 4]), page=rng.choice([128, 256]), vocab=32000, rows=256,
                gap=0.3, shape_seed=seed)


# ---- sizes of a case ---------------------------------------------------------------------------------------------
def _sizes(case):
    """(prefix lengths, tree sizes) of the batch: lengths log-uniform, trees uniform between the case's bounds."""
    rng = random.Random(case["shape_seed"])
    Ls = [case["l_lo"] if case["l_hi"] <= max(1, case["l_lo"]) else _log_int(rng, max(1, case["l_lo"]), case["l_hi"])
          for _ in range(case["n_req"])]
    ns = [rng.randint(case["n_lo"], case["n_hi"]) for _ in range(case["n_req"])]
    return Ls, ns


def _loop_prefix(case):
    return [case["l_lo"] + 3 * k + (k & 1) for k in range(case["steps"])]


def _attention_work(hq, hkv, d, Ls, ns, words):
    """K and V once, Q in, output out, mask rows; 4 D flops per visible pair and head (a tree row sees the prefix and
    its ancestors, about ln n of them)."""
    rows, n = sum(Ls) + sum(ns), sum(ns)
    pairs = sum(k * (L + 2 + math.log(k)) for L, k in zip(Ls, ns) if k)
    return 2 * rows * hkv * d * 2 + 2 * n * hq * d * 2 + n * words * 4, 4 * hq * d * pairs


def work(case):
    op = case["op"]
    if op == "attend":
        Ls, ns = _sizes(case)
        b, f = _attention_work(case["hq"], case["hkv"], case["d"], Ls, ns, B.dyspec_words_per_row(max(ns)))
        return {"bytes": b * case["layers"], "flops": f * case["layers"]}
    if op == "loop":
        W = B.dyspec_words_per_row(case["n_lo"])
        got = [_attention_work(case["hq"], case["hkv"], case["d"], [L], [case["n_lo"]], W) for L in _loop_prefix(case)]
        return {"bytes": sum(b for b, _ in got) * case["layers"], "flops": sum(f for _, f in got) * case["layers"]}
    if op == "verify":      # the draft and target row of the node where the walk ends, two numbers per node before it
        return {"bytes": case["n_req"] * 2 * case["vocab"] * 4 + 16 * case["n_req"] * case["n_hi"],
                "flops": case["n_req"] * 4 * case["vocab"]}
    if op == "grow":        # every table row that the trees can reach once; one sum over a row per guess
        guesses = case["n_req"] * case["m"]
        return {"bytes": min(guesses, case["rows"]) * case["vocab"] * 4 + guesses * 20, "flops": guesses * case["vocab"]}
    Ls, ns = _sizes(dict(case, n_lo=case["m"] + 1, n_hi=case["m"] + 1))
    b, f = _attention_work(case["hq"], case["hkv"], case["d"], Ls, ns, B.dyspec_words_per_row(case["m"] + 1))
    grown = case["n_req"] * case["m"]
    return {"bytes": b * case["layers"] + (min(grown, case["rows"]) + 2 * case["n_req"]) * case["vocab"] * 4,
            "flops": f * case["layers"] + grown * case["vocab"]}


def tolerance(case):
    # bf16 outputs, P rounded to bf16, sums in another order: the same calls under three other plans (other splits,
    # the other kernel) differ by rel 2.9e-3 and max 2.8e-2 at most
    if case["op"] in ("attend", "loop"):
        return {"rel": 1e-2, "max": 0.1}
    # token and node numbers; fp32 values of the trees (sums of a row in fp64).  A decision whose number lies within
    # rounding of its threshold may fall the other way, and then changes one request's walk.
    if case["op"] == "verify":
        return {"rel": 0.0, "differ": 0.005}
    if case["op"] == "grow":
        return {"rel": 1e-6, "max": 1e-5}
    return {"rel": 1e-2, "max": 0.1, "differ": 0.005}


# ---- the same results in 64 bits, in plain torch and numpy ------------------------------------------------------
def _ancestors(parents):
    """[n, n] truth values: row i sees itself and its ancestors."""
    see = np.eye(len(parents), dtype=bool)
    for i, p in enumerate(parents):
        if p >= 0:
            see[i] |= see[p]
    return see


def _preorder(parents):
    """Parent array after renumbering by a depth-first walk that takes children in index order."""
    children = [[] for _ in parents]
    for i, p in enumerate(parents):
        if p >= 0:
            children[p].append(i)
    todo, new = [i for i, p in enumerate(parents) if p < 0][::-1], {}
    while todo:
        i = todo.pop()
        new[i] = len(new)
        todo += children[i][::-1]
    out = np.zeros(len(parents), dtype=np.int64)
    for i, k in new.items():
        out[k] = new[parents[i]] if parents[i] >= 0 else -1
    return out


def _attention64(q, k, v, prefix_rows, tree_rows, see):
    """One request's tree attention: the prefix, then the tree's own rows under `see`."""
    g, rows = q.shape[1] // k.shape[1], torch.cat([prefix_rows, tree_rows])
    out = torch.empty(q.shape, dtype=torch.float64, device=DEV)
    hidden = torch.cat([torch.zeros((len(q), len(prefix_rows)), dtype=torch.bool, device=DEV), ~see], dim=1)
    for h in range(q.shape[1]):
        s = (q[:, h].double() @ k[rows, h // g].double().T) * q.shape[2] ** -0.5
        out[:, h] = torch.softmax(s.masked_fill_(hidden, -math.inf), dim=1) @ v[rows, h // g].double()
    return out


def _rows_of(case, Ls, ns, seed):
    """Per request: cache rows of the prefix tokens, cache rows of the tree."""
    ar, got = np.arange, []
    if case.get("layout") == "contiguous":
        first = [sum(Ls[:r]) + sum(ns[:r]) for r in range(len(Ls))]
        got = [(f + ar(L), f + L + ar(n)) for f, L, n in zip(first, Ls, ns)]
    else:
        page, inside = case["page"], case.get("layout") == "in_pages"
        table, tree0, _ = _pages(seed, Ls, ns, page, inside)
        for r, (L, n) in enumerate(zip(Ls, ns)):
            t = ar(L + n)
            at = table[r, t // page].astype(np.int64) * page + t % page
            got.append((at[:L], at[L:] if inside else tree0[r] + ar(n)))
    return [tuple(torch.from_numpy(x.astype(np.int64)).to(DEV) for x in pair) for pair in got]


def _batch64(case, s, seed, Ls, ns, parents):
    rows, offs, outs = _rows_of(case, Ls, ns, seed), np.concatenate([[0], np.cumsum(ns)]), []
    see = [torch.from_numpy(_ancestors(parents[offs[r]:offs[r + 1]])).to(DEV) for r in range(len(ns))]
    for q, k, v, _ in s["layers"]:
        outs.append(torch.cat([_attention64(q[offs[r]:offs[r + 1]], k, v, *rows[r], see[r]) for r in range(len(ns))]))
    return outs


def _grow64(case, s):
    """Algorithms 1 and 2 in fp64: value a node was drawn at, and value of the first draw under it."""
    T, V, U = case["rows"], case["vocab"], s["uniforms"].cpu().numpy()
    table, S = s["table"].cpu().numpy().astype(np.float64), case["m"] + 1
    values, childs = np.zeros((case["n_req"], S)), np.zeros((case["n_req"], S))
    parents = np.zeros((case["n_req"], S), dtype=np.int64)
    for r, root in enumerate(s["root"].cpu().numpy()):
        row, left, n = [int(root)], {}, 1
        values[r, 0] = childs[r, 0] = 1.0
        parents[r, 0] = -1

        def sample(pos, attempt, v):
            nonlocal n
            p = left.setdefault(pos, table[row[pos]].copy())
            cum = np.cumsum(p)
            y = min(int(np.searchsorted(cum, float(U[(row[pos] * 7919 + attempt * 104729 + 17) % len(U)]) * cum[-1], side="right")), V - 1)
            share = p[y] / cum[-1] if cum[-1] > 0 else 0.0
            p[y] = 0.0
            row.append(((row[pos] * 2654435761 + (y + 1) * 40503) % (1 << 32)) % T)
            parents[r, n], values[r, n], childs[r, n] = pos, v, v * share
            n += 1
            return share

        if case["algo"] == "greedy":
            heap, pushed = [(-1.0, 0, 0, 0)], 1
            while n < S and heap:
                v, _, pos, attempt = heapq.heappop(heap)
                share = sample(pos, attempt, -v)
                if 1.0 - share > 0.0:
                    heapq.heappush(heap, (v * (1.0 - share), pushed, pos, attempt + 1))
                heapq.heappush(heap, (v * share, pushed + 1, n - 1, 0))
                pushed += 2
        else:
            pos = 0
            while pos < n and n < S:
                v, attempt = childs[r, pos], 0
                while v >= np.float32(case["threshold"]) and n < S:
                    share = sample(pos, attempt, v)
                    v, attempt = v * (1.0 - share), attempt + 1
                    if not 1.0 - share > 0.0:
                        break
                left.pop(pos, None)
                pos += 1
    return parents, values, childs


def exact(case, seed):
    op = case["op"]
    if op == "verify":              # token and node numbers
        return None
    s = prepare(case, seed)
    if op == "grow":
        _, values, childs = _grow64(case, s)
        return [None, None, values, childs, None, None]
    if op == "attend":
        Ls, ns = _sizes(case)
        parents = s["parents"].cpu().numpy()
        if case["dfs"]:
            parents = _preorder(parents)
        return _batch64(case, s, seed, Ls, ns, parents) + [None] * (5 if case["dfs"] else 3)
    if op == "loop":
        outs, n = [], s["n"]
        for L, parents, _, layers in s["steps"]:
            see = torch.from_numpy(_ancestors(parents.cpu().numpy())).to(DEV)
            at = torch.arange(L + n, device=DEV)
            outs += [_attention64(q, k, v, at[:L], at[L:], see) for (q, _), (k, v) in zip(layers, s["caches"])]
        return outs
    parents, values, _ = _grow64(dict(case, algo="greedy", threshold=0.0), s)
    outs = [None, None, values] + [None] * 8
    for out in _batch64(case, s, seed, s["Ls"], s["ns"], parents.reshape(-1)):
        outs += [None, None, out]   # the cache after compaction: copies of its own rows
    return outs


# ---- set-up --------------------------------------------------------------------------------------------------------
def _gen(seed, k=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1009 + k)
    return g


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32).to(torch.bfloat16)


def _ints(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(DEV)


def _zeros(*shape, dtype=torch.int32):
    return torch.zeros(shape, dtype=dtype, device=DEV)


def _trees(seed, ns, alpha):
    """Best-first draft trees with Dirichlet(alpha) candidates; alpha 0: uniform random recursive trees."""
    rng = np.random.default_rng(seed)
    return [workloads.random_tree(rng, n) if alpha == 0.0 else workloads.greedy_tree(rng, n, 8, alpha) for n in ns]


def _pages(seed, Ls, ns, page, in_pages):
    """Shuffled page table, first tree row of each request (None: inside the pages), rows of the pool."""
    need = [-(-(L + n) // page) for L, n in zip(Ls, ns)]
    ids = np.random.default_rng(seed).permutation(sum(need))
    table = np.zeros((len(Ls), max(need)), dtype=np.int32)
    at = 0
    for r, k in enumerate(need):
        table[r, :k] = ids[at:at + k]
        at += k
    rows = sum(need) * page
    if in_pages:
        return table, None, rows
    tree0 = [rows + sum(ns[:r]) for r in range(len(ns))]
    return table, tree0, rows + sum(ns)


def _prepare_attend(case, seed):
    Ls, ns = _sizes(case)
    hq, hkv, d = case["hq"], case["hkv"], case["d"]
    n, W = sum(ns), B.dyspec_words_per_row(max(ns))
    s = dict(case=case, n=n, parents=_ints(np.concatenate(_trees(seed, ns, case["alpha"]))), bits=_zeros(n, W),
             depths=_zeros(n), status=_zeros(1), tiles=None, table=None)
    if case["layout"] == "contiguous":
        first = [sum(Ls[:r]) + sum(ns[:r]) for r in range(len(Ls))]
        rows = sum(Ls) + n
        s["plan"] = B.Plan(hq, hkv, d, Ls, ns, first, rows, W, 0.0)
    else:
        table, tree0, rows = _pages(seed, Ls, ns, case["page"], case["layout"] == "in_pages")
        s["plan"] = B.Plan(hq, hkv, d, Ls, ns, tree0, rows, W, 0.0, page_size=case["page"])
        s["table"], s["per_req"] = _ints(table), table.shape[1]
    if case["dfs"]:
        s["tiles"], s["new_parents"], s["order"] = _zeros(n), _zeros(n), _zeros(n)
    s["workspace"] = _zeros(max(256, s["plan"].workspace_bytes()), dtype=torch.uint8)
    g = _gen(seed)
    s["layers"] = [(_normal(g, n, hq, d), _normal(g, rows, hkv, d), _normal(g, rows, hkv, d),
                    torch.zeros((n, hq, d), dtype=torch.bfloat16, device=DEV)) for _ in range(case["layers"])]
    return s


def _run_attend(s):
    plan, bits, tiles, status, ws = s["plan"], s["bits"], s["tiles"], s["status"], s["workspace"]
    if tiles is not None:
        B.dyspec_plan_dfs_reorder(plan, s["parents"], s["order"], None, s["new_parents"], status)
        B.dyspec_plan_build_tree_mask_tiles(plan, s["new_parents"], bits, s["depths"], tiles, status)
    else:
        B.dyspec_plan_build_tree_mask(plan, s["parents"], bits, s["depths"], status)
    for q, k, v, out in s["layers"]:
        if s["table"] is not None:
            B.dyspec_tree_attention_paged(plan, q, k, v, s["table"], s["per_req"], bits, None, out, ws, status)
        elif tiles is not None:
            B.dyspec_tree_attention_ragged_sparse(plan, q, k, v, bits, tiles, out, ws, None, status)
        else:
            B.dyspec_tree_attention_ragged(plan, q, k, v, bits, out, ws, None, status)
    outs = [layer[3] for layer in s["layers"]] + [bits, s["depths"], status]
    return outs + [s["order"], tiles] if tiles is not None else outs


def _prepare_loop(case, seed):
    hq, hkv, d, n = case["hq"], case["hkv"], case["d"], case["n_lo"]
    W = B.dyspec_words_per_row(n)
    rows = _loop_prefix(case)[-1] + n
    g = _gen(seed)
    trees = _trees(seed, [n] * case["steps"], case["alpha"])
    s = dict(case=case, n=n, W=W, caches=[(_normal(g, rows, hkv, d), _normal(g, rows, hkv, d)) for _ in range(case["layers"])],
             status=_zeros(1), steps=[])
    for L, tree in zip(_loop_prefix(case), trees):
        s["steps"].append((L, _ints(tree), _zeros(n, W), [(_normal(g, n, hq, d), torch.zeros((n, hq, d), dtype=torch.bfloat16, device=DEV))
                                                          for _ in range(case["layers"])]))
    B.dyspec_set_default_shape(hq, hkv, d, W, 0.0)
    return s


def _run_loop(s):
    n, W = s["n"], s["W"]
    for L, parents, bits, layers in s["steps"]:
        B.dyspec_build_tree_mask(parents, n, bits, None, W, s["status"])
        for (q, out), (k, v) in zip(layers, s["caches"]):
            B.dyspec_tree_attention(q, k, v, L, bits, n, out)
    return [out for _, _, _, layers in s["steps"] for _, out in layers]


def _softmax_rows(x):
    return torch.softmax(x, dim=1)


def _prepare_verify(case, seed):
    _, ns = _sizes(dict(case, l_lo=0, l_hi=0))
    N, V = sum(ns), case["vocab"]
    trees = _trees(seed, ns, 0.3)
    g = _gen(seed)
    logits = 3.0 * torch.randn((N, V), generator=g, device=DEV)
    draft = _softmax_rows(logits)
    target = _softmax_rows(logits + case["gap"] * torch.randn((N, V), generator=g, device=DEV))
    # a node's children carry tokens drawn from its draft row without replacement, in order (Gumbel top-k)
    offs = np.concatenate([[0], np.cumsum(ns)])
    rank = np.zeros(N, dtype=np.int64)
    owner = np.zeros(N, dtype=np.int64)
    for r, tree in enumerate(trees):
        seen = np.zeros(len(tree), dtype=np.int64)
        for i in range(1, len(tree)):
            rank[offs[r] + i], owner[offs[r] + i] = seen[tree[i]], offs[r] + tree[i]
            seen[tree[i]] += 1
    gumbel = -torch.log(-torch.log(torch.rand((N, V), generator=g, device=DEV).clamp_(1e-12, 1.0 - 1e-7)))
    best = torch.topk(logits + gumbel, min(V, int(rank.max()) + 1), dim=1).indices
    tokens = best[torch.from_numpy(owner).to(DEV), torch.from_numpy(rank).to(DEV)].to(torch.int32)
    u = torch.rand((2, N), generator=g, device=DEV)
    return dict(case=case, parents=_ints(np.concatenate(trees)), tokens=tokens.contiguous(), draft=draft.contiguous(),
                target=target.contiguous(), accept=u[0].contiguous(), sample=u[1].contiguous(), offs=_ints(offs), max_nodes=max(ns),
                out_tokens=_zeros(case["n_req"], 64), out_nodes=_zeros(case["n_req"], 64), count=_zeros(case["n_req"]), status=_zeros(1))


def _run_verify(s):
    c = s["case"]
    B.dyspec_verify_tree(s["parents"], s["tokens"], s["draft"], s["target"], s["accept"], s["sample"], s["offs"], c["n_req"],
                         s["max_nodes"], c["vocab"], s["out_tokens"], s["out_nodes"], s["count"], 64, c["bonus"], s["status"])
    return [s["out_tokens"], s["out_nodes"], s["count"], s["status"]]


def _draft_table(g, rows, vocab):
    """Language-model-like rows: p ~ rank^-a over shuffled tokens, a between 1.1 and 2.2."""
    a = 1.1 + 1.1 * torch.rand((rows, 1), generator=g, device=DEV)
    p = torch.arange(1, vocab + 1, device=DEV, dtype=torch.float32)[None, :] ** -a
    p /= p.sum(dim=1, keepdim=True)
    order = torch.argsort(torch.rand((rows, vocab), generator=g, device=DEV), dim=1)
    return torch.zeros_like(p).scatter_(1, order, p).contiguous()


def _prepare_grow(case, seed):
    g = _gen(seed)
    R, S = case["n_req"], case["m"] + 1
    return dict(case=case, table=_draft_table(g, case["rows"], case["vocab"]), uniforms=torch.rand(4099, generator=g, device=DEV),
                root=torch.randint(0, case["rows"], (R,), generator=g, device=DEV, dtype=torch.int32),
                parents=_zeros(R, S), tokens=_zeros(R, S), values=_zeros(R, S, dtype=torch.float32),
                child_values=_zeros(R, S, dtype=torch.float32), rows=_zeros(R, S), count=_zeros(R))


def _run_grow(s):
    c = s["case"]
    outs = [s["parents"], s["tokens"], s["values"], s["child_values"], s["rows"], s["count"]]
    if c["algo"] == "greedy":
        B.dyspec_build_tree_greedy(s["table"], c["rows"], c["vocab"], s["uniforms"], 4099, s["root"], c["n_req"], c["m"], *outs)
    else:
        B.dyspec_build_tree_threshold(s["table"], c["rows"], c["vocab"], s["uniforms"], 4099, s["root"], c["n_req"],
                                      c["threshold"], c["m"], *outs)
    return outs


def _prepare_decode(case, seed):
    n_req, n = case["n_req"], case["m"] + 1
    hq, hkv, d, V = case["hq"], case["hkv"], case["d"], case["vocab"]
    Ls, ns = _sizes(dict(case, n_lo=n, n_hi=n))
    s = _prepare_grow(dict(case, algo="greedy", threshold=0.0), seed)
    _run_grow(s)                                 # the draft rows of the nodes that the step's tree will have
    g = _gen(seed, 1)
    s["draft"] = s["table"][s["rows"].reshape(-1).long()].contiguous()
    s["target"] = s["draft"] * torch.exp(case["gap"] * torch.randn((n_req * n, V), generator=g, device=DEV))
    s["target"] /= s["target"].sum(dim=1, keepdim=True)
    u = torch.rand((2, n_req * n), generator=g, device=DEV)
    table, tree0, rows = _pages(seed, Ls, ns, case["page"], False)
    W = B.dyspec_words_per_row(n)
    s.update(case=case, Ls=Ls, ns=ns, W=W, pool=rows, tree0=tree0, tree0_dev=torch.tensor(tree0, dtype=torch.int64, device=DEV),
             pages=_ints(table), per_req=table.shape[1], prefix=_ints(Ls), offs=_ints(np.arange(n_req + 1) * n), accept=u[0].contiguous(),
             sample=u[1].contiguous(), bits=_zeros(n_req * n, W), depths=_zeros(n_req * n), status=_zeros(1),
             out_tokens=_zeros(n_req, 64), out_nodes=_zeros(n_req, 64), emitted=_zeros(n_req), new_prefix=_zeros(n_req))
    s["layers"] = [(_normal(g, n_req * n, hq, d), _normal(g, rows, hkv, d), _normal(g, rows, hkv, d),
                    torch.zeros((n_req * n, hq, d), dtype=torch.bfloat16, device=DEV)) for _ in range(case["layers"])]
    return s


def _run_decode(s):
    c = s["case"]
    n_req, n, page = c["n_req"], c["m"] + 1, c["page"]
    B.dyspec_build_tree_greedy(s["table"], c["rows"], c["vocab"], s["uniforms"], 4099, s["root"], n_req, c["m"], s["parents"],
                               s["tokens"], s["values"], s["child_values"], s["rows"], s["count"])
    plan = B.Plan(c["hq"], c["hkv"], c["d"], s["Ls"], s["ns"], s["tree0"], s["pool"], s["W"], 0.0, page_size=page)
    ws = torch.zeros(max(256, plan.workspace_bytes()), dtype=torch.uint8, device=DEV)
    B.dyspec_plan_build_tree_mask(plan, s["parents"], s["bits"], s["depths"], s["status"])
    for q, k, v, out in s["layers"]:
        B.dyspec_tree_attention_paged(plan, q, k, v, s["pages"], s["per_req"], s["bits"], None, out, ws, s["status"])
    B.dyspec_verify_tree(s["parents"], s["tokens"], s["draft"], s["target"], s["accept"], s["sample"], s["offs"], n_req, n, c["vocab"],
                         s["out_tokens"], s["out_nodes"], s["emitted"], 64, True, s["status"])
    for _, k, v, _ in s["layers"]:
        B.dyspec_compact_kv_paged(k, v, s["tree0_dev"], s["pages"], s["per_req"], page, s["prefix"], s["out_nodes"], s["emitted"],
                                  n_req, 64, c["hkv"], c["d"], s["new_prefix"], s["status"], keep_root=True)
    plan.destroy()
    outs = [s[k] for k in ("parents", "tokens", "values", "rows", "bits", "depths", "out_tokens", "out_nodes", "emitted", "new_prefix", "status")]
    return outs + [t for layer in s["layers"] for t in layer[1:]]


_PREPARE = dict(attend=_prepare_attend, loop=_prepare_loop, verify=_prepare_verify, grow=_prepare_grow, decode=_prepare_decode)
_RUN = dict(attend=_run_attend, loop=_run_loop, verify=_run_verify, grow=_run_grow, decode=_run_decode)


def prepare(case, seed):
    return _PREPARE[case["op"]](case, seed)


def run(state):
    return _RUN[state["case"]["op"]](state)
