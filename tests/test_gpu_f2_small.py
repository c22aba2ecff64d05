"""Two-float RKC of the smallest states: one to five species, whose state
lives in registers (up to three) or in shared-memory rows.  Up to three
species no proposal network and no joined estimates: the work queue gives
the static mapping's results bit for bit, and every form is within the
two-float bar of the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1611_02274_gb300 import binding as B
from paper_1611_02274_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def network(species, nsys):
    rng = np.random.default_rng(species)
    y0 = rng.uniform(0.1, 1.0, (species, nsys))
    net = W.make_network(11, species, 2 * species + 1)
    return W.Workload("network", W.RHS_MASSACTION, W.METHOD_RKC, nsys, species, np.ascontiguousarray(y0 / y0.sum(axis=0)),
                      rng.uniform(1000.0, 2000.0, (1, nsys)), 0.0, 2e-5, 1e-7, 1e-12, network=net)


def run(w, prec, mapping):
    import torch
    h = B.register_workload(w)
    cnt = B.counters_like(w.nsys, "cuda")
    y = B.integrate("rkc", h, torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda(), w.t0, w.tend, w.rtol,
                    w.atol, counters=cnt, precision=prec, mapping=mapping, sync=True).cpu().numpy()
    B.release(h)
    return y, cnt.n_rhs.cpu().numpy(), cnt.n_accept.cpu().numpy()


@pytest.mark.parametrize("prec", [B.ODE_PREC_F2, B.ODE_PREC_F2_LEAN])
@pytest.mark.parametrize("species", [1, 2, 3, 4, 5])
def test_small_networks(species, prec):
    w = network(species, 301)
    w.tend, w.rtol = 1e-6, 1e-6
    ref = O.integrate(O.model_for(w), W.METHOD_RKC, w.y0, w.params, w.t0, w.tend, w.rtol, w.atol)
    for mapping in (B.ODE_MAP_THREAD, B.ODE_MAP_QUEUE):
        y = run(w, prec, mapping)[0]
        assert (np.abs(y - ref.y) / (np.abs(ref.y) + w.atol)).max() <= 1e-5  # the two-float form's bar


@pytest.mark.parametrize("prec", [B.ODE_PREC_F2, B.ODE_PREC_F2_LEAN])
@pytest.mark.parametrize("species", [2, 3])
def test_no_joined_estimates_up_to_three_species(species, prec):
    w = network(species, 301)
    y, n_rhs, n_acc = run(w, prec, B.ODE_MAP_THREAD)
    assert n_acc.max() > 100  # several estimates of the spectral radius
    q = run(w, prec, B.ODE_MAP_QUEUE)
    np.testing.assert_array_equal(q[0], y)
    np.testing.assert_array_equal(q[1], n_rhs)
