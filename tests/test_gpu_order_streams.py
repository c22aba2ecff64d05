"""The automatic parameter order and the calls around it: its memory belongs
to one call, so neither a captured graph of a cost-ordered call, nor another
stream, nor a second thread whose per-thread stream has the same handle
value, sees it.  Results are compared bit for bit with the same batch in its
own order (a capturing-size batch below the order's threshold gives each
system's own result: systems are independent)."""
import ctypes
import threading

import numpy as np
import pytest

from paper_1611_02274_gb300 import binding as B
from paper_1611_02274_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PER_THREAD = 2  # cudaStreamPerThread: one handle value, a stream in every thread


def device(w):
    import torch
    return torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda()


def call(h, w, y0, p, y, cnt, stream, **kw):
    return B.integrate("rkck", h, y0, p, w.t0, w.tend, w.rtol, w.atol, y_out=y, counters=cnt,
                       mapping=B.ODE_MAP_THREAD, stream=stream, **kw)


def in_pieces(h, w, y0, p):
    """The batch in pieces too small to be ordered."""
    import torch
    ys, ns = [], []
    for k in range(0, w.nsys, 4000):
        a, b = y0[:, k:k + 4000].contiguous(), p[:, k:k + 4000].contiguous()
        cnt = B.counters_like(a.shape[1], "cuda")
        ys.append(call(h, w, a, b, torch.empty_like(a), cnt, None, sync=True))
        assert not B.last_launch()["ordered"]
        ns.append(cnt.n_rhs)
    return torch.cat(ys, dim=1).cpu().numpy(), torch.cat(ns).cpu().numpy()


def test_graph_of_a_cost_ordered_call_survives_larger_calls():
    """Capture a call with a cost, run a larger batch without one on the same stream, replay."""
    import torch
    small, large = W.vdp(30000, seed=1), W.vdp(90000, seed=2)
    h = B.register_workload(small)
    y0, p = device(small)
    ly0, lp = device(large)
    ref_y, ref_n = in_pieces(h, small, y0, p)
    lref_y, lref_n = in_pieces(h, large, ly0, lp)
    cost = torch.from_numpy(ref_n.astype(np.float32)).cuda()
    y, cnt = torch.empty_like(y0), B.counters_like(small.nsys, "cuda")
    ly, lcnt = torch.empty_like(ly0), B.counters_like(large.nsys, "cuda")
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(s):
        call(h, small, y0, p, y, cnt, s.cuda_stream, cost=cost)  # buffers of the cost order
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            call(h, small, y0, p, y, cnt, s.cuda_stream, cost=cost)
    for _ in range(3):
        y.zero_()
        cnt.n_rhs.zero_()
        torch.cuda.synchronize()
        call(h, large, ly0, lp, ly, lcnt, s.cuda_stream)         # beside the replay
        assert B.last_launch()["ordered"]
        with torch.cuda.stream(other):
            g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(y.cpu().numpy(), ref_y)
        np.testing.assert_array_equal(cnt.n_rhs.cpu().numpy(), ref_n)
        np.testing.assert_array_equal(ly.cpu().numpy(), lref_y)
        np.testing.assert_array_equal(lcnt.n_rhs.cpu().numpy(), lref_n)
    B.release(h)


@pytest.mark.parametrize("stream", ["per_thread", "own"])
def test_threads_keep_their_orders_apart(stream):
    """Two host threads at once, on the per-thread stream's one handle value and on streams of their own."""
    import torch
    ws = [W.vdp(40000, seed=3), W.vdp(30011, seed=4)]
    h = B.register_workload(ws[0])
    dev = [device(w) for w in ws]
    refs = [in_pieces(h, w, *d) for w, d in zip(ws, dev)]
    outs = [[(torch.zeros_like(d[0]), B.counters_like(w.nsys, "cuda")) for _ in range(8)] for w, d in zip(ws, dev)]
    streams = [PER_THREAD if stream == "per_thread" else torch.cuda.Stream().cuda_stream for _ in ws]
    torch.cuda.synchronize()
    ordered = [[], []]
    gate = threading.Barrier(2)

    def work(t):
        gate.wait()
        for y, cnt in outs[t]:
            call(h, ws[t], *dev[t], y, cnt, ctypes.c_void_p(streams[t]).value)
            ordered[t].append(B.last_launch()["ordered"])

    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert all(ordered[0]) and all(ordered[1])
    for t in range(2):
        for y, cnt in outs[t]:
            np.testing.assert_array_equal(y.cpu().numpy(), refs[t][0])
            np.testing.assert_array_equal(cnt.n_rhs.cpu().numpy(), refs[t][1])
    B.release(h)


def test_every_stream_is_ordered_and_capture_is_not():
    """The order does not depend on how many streams a program uses; a captured call takes the batch's own order."""
    import torch
    w = W.vdp(20011, seed=5)
    h = B.register_workload(w)
    y0, p = device(w)
    ref_y, _ = in_pieces(h, w, y0, p)
    streams = [torch.cuda.Stream() for _ in range(20)]
    outs = [torch.empty_like(y0) for _ in streams]
    cnt = B.counters_like(w.nsys, "cuda")
    torch.cuda.synchronize()
    for s, y in zip(streams, outs):
        call(h, w, y0, p, y, None, s.cuda_stream)
        assert B.last_launch()["ordered"]
    torch.cuda.synchronize()
    for y in outs:
        np.testing.assert_array_equal(y.cpu().numpy(), ref_y)
    s, y = streams[0], torch.empty_like(y0)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s), torch.cuda.graph(g, stream=s):
        call(h, w, y0, p, y, cnt, s.cuda_stream)
        assert not B.last_launch()["ordered"]
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(y.cpu().numpy(), ref_y)
    B.release(h)
