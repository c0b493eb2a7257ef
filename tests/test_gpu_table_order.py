"""The entry points without a plan send their work list down the stream in front of the attention launch.  That launch may only
start early where it reads nothing of the list before it waits, that is with one item a CTA (the first items travel with the
launch).  Seen in a captured graph: with several items a CTA all edges are full dependencies.  Run from the graph,
the output is that of the calls outside."""
import numpy as np
import pytest

from paper_2410_11744_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entry", ["static", "single"])
@pytest.mark.parametrize("L,n,several", [(200, 1024, True), (100, 2000, True), (1500, 40, False), (300, 6, False)])
def test_attention_waits_for_the_work_list_in_front_of_it(entry, L, n, several):
    import torch
    rt = pytest.importorskip("cuda.bindings.runtime")
    from paper_2410_11744_b200 import build
    build.build()
    from paper_2410_11744_b200 import binding as B, runner as R
    hq, hkv, d = 64, 8, 128
    b = R.DeviceBatch(wl.make_custom(L + n, hq, hkv, d, [L], [wl.greedy_tree(np.random.default_rng(n), n, 8, 0.3)]))
    b.step()
    want, out = torch.zeros_like(b.out), torch.zeros_like(b.out)
    B.dyspec_tree_attention_static(b.q, b.k, b.v, L, b.bits, n, want, hq, hkv, d, b.W)
    torch.cuda.synchronize()
    assert (want.float() - b.out.float()).abs().max() <= 2e-2            # (the plan's own call may split the work differently)
    stream = torch.cuda.Stream()
    h = stream.cuda_stream
    B.dyspec_release_cache()
    B.dyspec_set_default_shape(hq, hkv, d, b.W, 0.0)
    for k in range(1, 9):                                                # the memory of all eight slots; the size itself stays new
        B.dyspec_tree_attention(b.q, b.k, b.v, L - k, b.bits, n, out, stream=h)
    stream.synchronize()

    assert rt.cudaStreamBeginCapture(h, rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed)[0] == 0
    if entry == "static":
        B.dyspec_tree_attention_static(b.q, b.k, b.v, L, b.bits, n, out, hq, hkv, d, b.W, stream=h)
    else:
        B.dyspec_tree_attention(b.q, b.k, b.v, L, b.bits, n, out, stream=h)
    err, graph = rt.cudaStreamEndCapture(h)
    assert err == 0
    err, *_, count = rt.cudaGraphGetEdges(graph)
    assert err == 0 and count >= 1 and not b.plan.describe()["combine_launch"]      # (a combine kernel would start early)
    full = rt.cudaGraphGetEdges(graph, count)[0] == 0                    # "lossy" where an edge is not a full dependency
    assert full == several
    err, run = rt.cudaGraphInstantiate(graph, 0)
    assert err == 0
    for _ in range(2):
        out.zero_()
        torch.cuda.synchronize()
        assert rt.cudaGraphLaunch(run, h)[0] == 0
        stream.synchronize()
        assert torch.equal(out, want)
    rt.cudaGraphExecDestroy(run)
    rt.cudaGraphDestroy(graph)
    B.dyspec_release_cache()
