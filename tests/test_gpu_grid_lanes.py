"""Lanes per system and threads per block of the plain FP64 form, at both
sides of each line of the rule (in rounds of warps, so from the device's SM
count), with the oracle's results bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1611_02274_gb300 import binding as B
from paper_1611_02274_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def slots():
    import torch
    return 4 * torch.cuda.get_device_properties(0).multi_processor_count


def make(family, points, nsys, tend):
    if family == "bruss":
        w = W.bruss(nsys=nsys, n=points, seed=points)
        w.tend = tend
        return w
    rng = np.random.default_rng(points)
    return W.Workload("chain", W.RHS_VDP_CHAIN, W.METHOD_RKCK, nsys, 2 * points,
                      rng.uniform(-2.0, 2.0, (2 * points, nsys)), 10.0 ** rng.uniform(-1.0, 1.0, (1, nsys)), 0.0, tend,
                      1e-6, 1e-9)


def run(w, method, cost=None):
    import torch
    h = B.register_workload(w)
    cnt = B.counters_like(w.nsys, "cuda")
    c = None if cost is None else torch.from_numpy(cost).cuda()
    y = B.integrate(method, h, torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda(), w.t0, w.tend, w.rtol,
                    w.atol, counters=cnt, mapping=B.ODE_MAP_THREAD, cost=c, sync=True).cpu().numpy()
    info = B.last_launch()
    B.release(h)
    r = O.integrate(O.model_for(w), {"rkck": W.METHOD_RKCK, "rkc": W.METHOD_RKC}[method], w.y0, w.params, w.t0, w.tend,
                    w.rtol, w.atol)
    np.testing.assert_array_equal(y, r.y)
    np.testing.assert_array_equal(cnt.n_rhs.cpu().numpy(), r.n_rhs)
    return info


# family, method, points, lanes where narrow, rounds of warps (a warp per system) from which unordered batches are narrow
@pytest.mark.parametrize("family,method,points,lanes,rounds", [
    ("bruss", "rkc", 4, 1, 4), ("bruss", "rkc", 32, 8, 4), ("bruss", "rkc", 64, 16, 4),
    ("bruss", "rkck", 5, 2, 4), ("bruss", "rkck", 16, 4, 4), ("chain", "rkc", 16, 4, 8), ("chain", "rkck", 8, 2, 11)])
def test_lanes_by_size(family, method, points, lanes, rounds):
    for nsys, want in ((rounds * slots() - 1, 32), (rounds * slots(), lanes)):
        info = run(make(family, points, nsys, 0.002), method)
        assert info["lanes"] == want and not info["ordered"], (nsys, info)


@pytest.mark.parametrize("family,method,points,lanes,narrow", [("bruss", "rkck", 24, 8, 2.0), ("bruss", "rkck", 48, 16, 2.0),
                                                               ("chain", "rkc", 32, 8, 2.0), ("chain", "rkck", 48, 16, 2.8)])
def test_wider_grids_are_narrow_in_order_only(family, method, points, lanes, narrow):
    n = int(np.ceil(narrow * 32 / lanes * slots()))
    w = make(family, points, n, 0.002)
    assert run(w, method)["lanes"] == 32                                            # short: not ordered
    assert run(w, method, cost=w.params[0].astype(np.float32))["lanes"] == lanes
    small = W.subset(w, np.arange(n - 32 // lanes - 1))
    assert run(small, method, cost=small.params[0].astype(np.float32))["lanes"] == 32


def test_one_warp_blocks():
    n = 32 * (slots() // 4)
    for nsys in (n, n + 1):  # both sides of an SM's count of blocks
        info = run(make("chain", 33, nsys, 0.002), "rkck")
        assert info["block"] == 32 and info["lanes"] == 32
