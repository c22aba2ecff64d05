"""When a batch is taken in parameter order, and which batches keep their own:
equal costs, parameters whose neighbours are alike already, short intervals
and small batches.  Results through the order are the oracle's, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1611_02274_gb300 import binding as B
from paper_1611_02274_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def order_of(p):
    import torch
    return B.parameter_order(torch.from_numpy(np.ascontiguousarray(p, dtype=np.float64)).cuda()).cpu().numpy()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 257, 20001, 300007])
def test_random_parameters_are_ordered_equal_ones_are_not(n):
    import torch
    rng = np.random.default_rng(n)
    p = 10.0 ** rng.uniform(-1.0, 1.0, n)
    idx = order_of(p)
    np.testing.assert_array_equal(np.sort(idx), np.arange(n))
    if n > 1000:  # classes are 1/65535 of the range of the float bits: neighbours may swap within one
        assert np.all(np.diff(np.log(p[idx])) < 2.0 * np.log(100.0) / 65535 * 1.5)
    same = np.arange(n, dtype=np.int32)
    for v in (3.7, 0.0, -1.0, np.nan, np.inf):
        np.testing.assert_array_equal(order_of(np.full(n, v)), same)
    for c in (torch.full((n,), 2.5, device="cuda"), torch.full((n,), 7, dtype=torch.int32, device="cuda")):
        np.testing.assert_array_equal(B.cost_order(c).cpu().numpy(), same)


def test_layouts_with_like_neighbours_are_kept():
    rng = np.random.default_rng(1)
    n = 40000
    p = rng.uniform(1000.0, 2000.0, n)
    smooth = 1500.0 + 500.0 * np.sin(np.arange(n) / 900.0)
    by_noisy_cost = p[np.argsort(p + rng.normal(0.0, 60.0, n))]
    for q in (np.sort(p), np.sort(p)[::-1], smooth, by_noisy_cost):
        np.testing.assert_array_equal(order_of(q), np.arange(n))
    assert np.all(np.diff(p[order_of(p)]) < 1.0)
    # a cost the caller gave is always followed, whatever the layout
    import torch
    idx = B.cost_order(torch.from_numpy(np.sort(p).astype(np.float32)).cuda()).cpu().numpy()
    assert idx[0] > n - 10


def test_special_parameters():
    rng = np.random.default_rng(2)
    p = rng.choice([np.nan, np.inf, -np.inf, 0.0, -3.0, 1e-310, 1e-40, 1.0, 2.0, 1e300], 20000)
    idx = order_of(p)
    np.testing.assert_array_equal(np.sort(idx), np.arange(p.size))
    with np.errstate(over="ignore"):
        f = p[idx].astype(np.float32)
    key = np.where(f > 0, f, 0.0)
    assert np.all(np.diff(key.view(np.uint32).astype(np.int64)) <= 0)


def run(w, method, prec=B.ODE_PREC_FP64, mapping=B.ODE_MAP_THREAD):
    import torch
    h = B.register_workload(w)
    cnt = B.counters_like(w.nsys, "cuda")
    y = B.integrate(method, h, torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda(), w.t0, w.tend, w.rtol,
                    w.atol, counters=cnt, precision=prec, mapping=mapping, sync=True).cpu().numpy()
    ordered = B.last_launch()["ordered"]
    B.release(h)
    return y, cnt, ordered


def make(kind, n, tend):
    w = {"vdp": lambda: W.vdp(n, seed=7), "mass": lambda: W.massaction(n, seed=7),
         "bruss": lambda: W.bruss(n, 32, seed=7)}[kind]()
    w.tend = tend
    return w


@pytest.mark.parametrize("kind,n,tend,method,prec", [
    ("vdp", 60000, 0.01, "rkck", B.ODE_PREC_FP64), ("vdp", 19000, 5.0, "rkck", B.ODE_PREC_FP64),
    ("vdp", 100000, 0.5, "rkck", B.ODE_PREC_MIXED_LEAN), ("vdp", 60000, 0.3, "rkc", B.ODE_PREC_F2_LEAN),
    ("mass", 20000, 1e-7, "rkc", B.ODE_PREC_MIXED_LEAN), ("mass", 20000, 1e-7, "rkc", B.ODE_PREC_F2_LEAN)])
def test_short_or_small_calls_keep_their_order(kind, n, tend, method, prec):
    assert not run(make(kind, n, tend), method, prec)[2]


@pytest.mark.parametrize("kind,n,tend,method", [("vdp", 40003, 1.0, "rkck"), ("vdp", 40003, 0.1, "rkc"),
                                                ("mass", 19501, 6e-6, "rkc"), ("bruss", 5003, 0.05, "rkc")])
def test_ordered_batches_are_the_oracles(kind, n, tend, method):
    w = make(kind, n, tend)
    y, cnt, ordered = run(w, method)
    assert ordered
    r = O.integrate(O.model_for(w), {"rkck": W.METHOD_RKCK, "rkc": W.METHOD_RKC}[method], w.y0, w.params, w.t0, w.tend,
                    w.rtol, w.atol)
    np.testing.assert_array_equal(y, r.y)
    np.testing.assert_array_equal(cnt.n_rhs.cpu().numpy(), r.n_rhs)


@pytest.mark.parametrize("prec", [B.ODE_PREC_F2_LEAN, B.ODE_PREC_MIXED])
def test_ordered_networks_are_the_unordered_ones(prec):
    w = make("mass", 30011, 1e-5)
    y, cnt, ordered = run(w, "rkc", prec)
    assert ordered
    for k in range(0, w.nsys, 10000):
        part = W.subset(w, np.arange(k, min(k + 10000, w.nsys)))
        yk, ck, o = run(part, "rkc", prec)
        assert not o
        np.testing.assert_array_equal(y[:, k:k + 10000], yk)
        np.testing.assert_array_equal(cnt.n_rhs.cpu().numpy()[k:k + 10000], ck.n_rhs.cpu().numpy())
