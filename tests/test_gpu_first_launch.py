"""Whether a call is accepted must not depend on the calls before it.  Sizes whose dynamic shared memory stays below 48 KB while
the kernel's static part takes it above, each as the first launch of a fresh process, against the oracle."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))

VERIFY = """
import numpy as np
import test_gpu_verify as T
from paper_2410_11744_b200 import binding as B, workloads as wl
from oracle import dyspec_oracle as orc
vocab, n_req, max_nodes = {vocab}, {n_req}, {max_nodes}
case = wl.make_verify_case(n_req, vocab, [wl.chain_tree(1 + r % 3) for r in range(n_req)], sharpness=2.0, disagreement=1.5)
out_t, out_n, cnt, status = T.run_gpu(B, case, max_nodes=max_nodes)
assert status == 0
right = 0
for r in range(n_req):
    sl = slice(case.node_offsets[r], case.node_offsets[r + 1])
    A, nodes, _ = orc.verify_tree(case.parents[r], case.tokens[r], case.draft_probs[sl], case.target_probs[sl], case.accept_u[sl], case.sample_u[sl])
    right += out_t[r, :cnt[r]].tolist() == A
assert right >= n_req - 1 - n_req // 25, right
"""

CONSTRUCT = """
import test_gpu_construct as T
from paper_2410_11744_b200 import binding as B, workloads as wl
from oracle import dyspec_oracle as orc
rows, uni = wl.make_draft_table({m}, {n_rows}, {vocab}, 2.0)
roots = [r % {n_rows} for r in range({n_req})]
got = T.run_gpu(B, rows, uni, roots, m={m})
for r in (0, {n_req} - 1):
    T.compare(got, r, orc.build_tree_greedy(rows, uni, {m}, root_row=roots[r]))
"""


@pytest.mark.parametrize("program", [
    VERIFY.format(vocab=32000, n_req=24, max_nodes=768), VERIFY.format(vocab=8192, n_req=80, max_nodes=500),
    VERIFY.format(vocab=32000, n_req=1, max_nodes=1400), VERIFY.format(vocab=4096, n_req=3, max_nodes=1638),
    CONSTRUCT.format(vocab=8192, n_rows=64, m=16, n_req=80), CONSTRUCT.format(vocab=8192, n_rows=256, m=25, n_req=40),
    CONSTRUCT.format(vocab=4096, n_rows=64, m=26, n_req=74), CONSTRUCT.format(vocab=8192, n_rows=24, m=200, n_req=40)],
    ids=["verify_24_of_768", "verify_80_of_500", "verify_1_of_1400", "verify_3_of_1638", "grow_80_of_16", "grow_40_of_25", "grow_74_of_26", "grow_40_of_200"])
def test_first_launch_of_a_process(program):
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(HERE), HERE]))
    r = subprocess.run([sys.executable, "-c", program], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]

CAPTURED = """
import numpy as np, torch
import cuda.bindings.runtime as rt
from paper_2410_11744_b200 import binding as B, workloads as wl
t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
case = wl.make_verify_case(3, 32000, [wl.chain_tree(3)] * 4, sharpness=2.0, disagreement=1.5)
par, tok, offs = t(np.concatenate(case.parents)), t(np.concatenate(case.tokens)), t(case.node_offsets)
dp, tp, au, su = t(case.draft_probs), t(case.target_probs), t(case.accept_u), t(case.sample_u)
rows, uni = wl.make_draft_table(5, 16, 4096, 2.0)
rows, uni, root = t(rows), t(uni), t(np.arange(4, dtype=np.int32))
outs = []
def call(stream):
    o = [torch.zeros((4, 64), dtype=torch.int32, device="cuda:0") for _ in range(5)] + [torch.zeros((4, 64), device="cuda:0") for _ in range(2)]
    c = [torch.zeros(4, dtype=torch.int32, device="cuda:0") for _ in range(2)]
    torch.cuda.synchronize()
    outs.append(o + c)
    return lambda: (B.dyspec_verify_tree(par, tok, dp, tp, au, su, offs, 4, 3, 32000, o[0], o[1], c[0], 64, bonus_at_leaf=True, stream=stream),
                    B.dyspec_build_tree_greedy(rows, 16, 4096, uni, len(uni), root, 4, 63, o[2], o[3], o[5], o[6], o[4], c[1], stream=stream))
s = torch.cuda.Stream()
h = s.cuda_stream
f = call(h)
assert rt.cudaStreamBeginCapture(h, rt.cudaStreamCaptureMode.cudaStreamCaptureModeGlobal)[0] == 0
f()
err, graph = rt.cudaStreamEndCapture(h)
assert err == 0, err
err, run = rt.cudaGraphInstantiate(graph, 0)
assert err == 0, err
assert rt.cudaGraphLaunch(run, h)[0] == 0
s.synchronize()
call(h)()
s.synchronize()
assert all(torch.equal(a, b) for a, b in zip(*outs)) and int(outs[0][8].min()) == 64
"""


def test_first_launch_inside_a_capture():
    pytest.importorskip("cuda.bindings.runtime")
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(HERE), HERE]))
    r = subprocess.run([sys.executable, "-c", CAPTURED], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
