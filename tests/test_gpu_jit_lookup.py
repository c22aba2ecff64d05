"""A launch finds its generated kernels by the network itself: networks that
differ in one constant keep their own kernels, and the lookup costs a call
little host time."""
import time

import numpy as np
import pytest

import oracle as O
from paper_1611_02274_gb300 import binding as B
from paper_1611_02274_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def run(w, prec):
    import torch
    h = B.register_workload(w)
    y = B.integrate("rkc", h, torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda(), w.t0, w.tend, w.rtol,
                    w.atol, precision=prec, sync=True).cpu().numpy()
    B.release(h)
    return y


def test_networks_that_differ_in_one_constant():
    w = W.massaction(40, seed=3, tend=1e-6)
    net = W.make_network(0)
    j = int(np.argmin(np.abs(net.log10A - net.Ea / (1500.0 * np.log(10.0)) - 4.0)))  # a rate inside the clip
    other = W.make_network(0)
    other.beta[j] += 0.25
    outs = []
    for nw in (net, other, net):
        w.network = nw
        ref = O.integrate(O.model_for(w), W.METHOD_RKC, w.y0, w.params, w.t0, w.tend, w.rtol, w.atol).y
        y = run(w, B.ODE_PREC_FP64)
        np.testing.assert_array_equal(y, ref)
        outs.append((y, run(w, B.ODE_PREC_F2_LEAN)))
    assert (outs[0][0] != outs[1][0]).any() and (outs[0][1] != outs[1][1]).any()
    np.testing.assert_array_equal(outs[0][1], outs[2][1])


@pytest.mark.parametrize("prec", [B.ODE_PREC_MIXED_LEAN, B.ODE_PREC_F2_LEAN])
def test_host_time_of_a_call(prec):
    """A call's host work is its launches: a tenth of a millisecond is ten times what they take."""
    import torch
    w = W.massaction(100, seed=3, tend=1e-9)
    h = B.register_workload(w)
    y0, p = torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda()
    y, t = torch.empty_like(y0), []
    for _ in range(60):
        a = time.perf_counter()
        B.integrate("rkc", h, y0, p, w.t0, w.tend, w.rtol, w.atol, y_out=y, precision=prec)
        t.append(time.perf_counter() - a)
        torch.cuda.synchronize()
    B.release(h)
    assert sorted(t)[len(t) // 2] < 1e-4, sorted(t)[:5]
