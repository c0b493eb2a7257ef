"""A plan's device tables are taken from a pool of the memory of plans destroyed before: a plan that is destroyed while its
kernels are still queued must keep its tables until they have run, whatever the stream, and later plans of other
shapes that take over its memory must not disturb them."""
import numpy as np
import pytest

from paper_2410_11744_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def test_plans_destroyed_with_their_kernels_still_queued():
    import torch
    assert torch.cuda.is_available()
    from paper_2410_11744_b200 import build
    build.build()
    from paper_2410_11744_b200 import binding as B, runner as R

    rng = np.random.default_rng(5)
    shapes = [([700, 33], [40, 8]), ([1500], [90]), ([64, 900, 257], [20, 64, 100]), ([300], [16])]   # both regimes, 16 KB tables and larger
    kept = [R.DeviceBatch(wl.make_custom(40 + i, 8, 2, 128, Ls, [wl.greedy_tree(rng, n, 6, 0.3) for n in ns]))
            for i, (Ls, ns) in enumerate(shapes)]
    for b in kept:
        b.step()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    spin = torch.zeros(1 << 26, device="cuda:0")
    rounds = []
    for k in range(60):                                     # several times the pool's bound
        b = kept[k % len(kept)]
        w = b.w
        with torch.cuda.stream(streams[k % 3]):
            if k % 7 == 0:
                spin.add_(1.0)                               # something to queue behind
            plan = B.Plan(w.n_q_heads, w.n_kv_heads, w.head_dim, w.prefix_len, w.n_nodes, w.kv_row_offset, b.kv_total_rows, b.W, 0.0)
            ws = torch.zeros(max(256, plan.workspace_bytes()), dtype=torch.uint8, device="cuda:0")
            out, bits = torch.zeros_like(b.out), torch.zeros_like(b.bits)
            B.dyspec_plan_build_tree_mask(plan, b.parents, bits, None, b.status)
            B.dyspec_tree_attention_ragged(plan, b.q, b.k, b.v, bits, out, ws, ws.numel(), b.status)
            plan.destroy()
        rounds.append((b, ws, bits, out))
    torch.cuda.synchronize()
    for b, _, bits, out in rounds:
        assert int(b.status.item()) == 0
        assert torch.equal(bits, b.bits) and torch.equal(out, b.out)
    B.dyspec_release_cache()
    again = R.DeviceBatch(kept[0].w)                         # the pool starts over
    again.step()
    torch.cuda.synchronize()
    assert torch.equal(again.out, kept[0].out)


def test_plans_created_while_the_cache_is_released():
    """A thread that gives everything back must not take the upload stream from another one's plan creation."""
    import threading
    import torch
    from paper_2410_11744_b200 import build
    build.build()
    from paper_2410_11744_b200 import binding as B, runner as R

    b = R.DeviceBatch(wl.make_custom(3, 8, 2, 128, [700, 33], [wl.greedy_tree(np.random.default_rng(3), n, 6, 0.3) for n in (40, 8)]))
    b.step()
    torch.cuda.synchronize()
    w, failed = b.w, []

    def create():
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(60):
                    plan = B.Plan(w.n_q_heads, w.n_kv_heads, w.head_dim, w.prefix_len, w.n_nodes, w.kv_row_offset, b.kv_total_rows, b.W, 0.0)
                    bits = torch.zeros_like(b.bits)
                    B.dyspec_plan_build_tree_mask(plan, b.parents, bits)
                    plan.destroy()
                    stream.synchronize()
                    assert torch.equal(bits, b.bits)
        except Exception as e:                               # noqa: BLE001  (reported by the main thread)
            failed.append(e)

    threads = [threading.Thread(target=create) for _ in range(3)]
    for t in threads:
        t.start()
    while any(t.is_alive() for t in threads):
        B.dyspec_release_cache()
    assert not failed, failed


def _tiny_plans(B, count):
    return [B.Plan(4, 4, 64, [10], [4], [0], 14, 4, 0.0) for _ in range(count)]


def test_memory_is_reused_only_after_a_wait_for_the_device():
    """Sixteen destructions behind a queued kernel, on a stream that waits for no other: by then the device has been waited for."""
    import torch
    from paper_2410_11744_b200 import build
    build.build()
    from paper_2410_11744_b200 import binding as B
    B.dyspec_release_cache()
    plans = _tiny_plans(B, 16)
    stream, done = torch.cuda.Stream(), torch.cuda.Event()
    x = torch.zeros(1 << 28, device="cuda:0")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for _ in range(100):                                 # some 30 ms
            x.add_(1.0)
        done.record()
    assert not done.query()
    for p in plans:
        p.destroy()
    assert done.query()
    B.dyspec_release_cache()


@pytest.mark.parametrize("mode", ["Global", "ThreadLocal", "Relaxed"])
def test_destruction_leaves_a_capture_alone(mode):
    """Plans are destroyed when Python collects them, in the middle of a stream capture too: the capture goes on, and what was
    to be waited for is used again afterwards."""
    import torch
    rt = pytest.importorskip("cuda.bindings.runtime")
    from paper_2410_11744_b200 import build
    build.build()
    from paper_2410_11744_b200 import binding as B
    B.dyspec_release_cache()
    plans, x = _tiny_plans(B, 40), torch.ones(1024, device="cuda:0")
    stream = torch.cuda.Stream()
    h = stream.cuda_stream
    torch.cuda.synchronize()
    assert rt.cudaStreamBeginCapture(h, getattr(rt.cudaStreamCaptureMode, "cudaStreamCaptureMode" + mode))[0] == 0
    for p in plans:
        p.destroy()
    assert rt.cudaMemsetAsync(x.data_ptr(), 0, 4096, h)[0] == 0
    err, graph = rt.cudaStreamEndCapture(h)
    assert err == 0
    rt.cudaGraphDestroy(graph)
    for p in _tiny_plans(B, 20):
        p.destroy()
    B.dyspec_release_cache()
