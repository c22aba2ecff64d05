"""The plain FP64 kernels' own arrangements of the method against the oracle,
bit for bit, at the sizes where an arrangement changes: kinetics mechanisms
from a few species to the largest, divisors outside the range that
quotients by reciprocal take, n-body rings, and the lanes a grid system takes."""
import numpy as np
import pytest

import oracle as O
from paper_1611_02274_gb300 import binding as B
from paper_1611_02274_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def assert_same(w, method, **kw):
    import torch
    h = B.register_workload(w)
    try:
        cnt = B.counters_like(w.nsys, "cuda")
        y = B.integrate(method, h, torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda(), w.t0, w.tend,
                        w.rtol, w.atol, counters=cnt, sync=True, **kw).cpu().numpy()
    finally:
        B.release(h)
    r = O.integrate(O.model_for(w), {"rkck": W.METHOD_RKCK, "rkc": W.METHOD_RKC}[method], w.y0, w.params, w.t0, w.tend,
                    w.rtol, w.atol)
    np.testing.assert_array_equal(cnt.n_accept.cpu().numpy(), r.n_accept)
    np.testing.assert_array_equal(cnt.n_rhs.cpu().numpy(), r.n_rhs)
    np.testing.assert_array_equal(y, r.y)


@pytest.mark.parametrize("species,reactions,density", [(12, 9, 1.0), (32, 33, 1.0), (33, 100, 1.0), (57, 766, 1.0),
                                                       (62, 1000, 1.0), (57, 766, 1e-31)])
def test_kinetics_sizes(species, reactions, density):
    """Mechanisms around a warp's 32 lanes; a density below 2^-100 divides in full."""
    mech = W.make_mechanism(3, species, reactions)
    rng = np.random.default_rng(species + reactions)
    n = 7
    Y = rng.uniform(0.0, 1.0, (species, n)) * (rng.random((species, n)) < 0.6)  # absent species are exact zeros
    Y[-1] += 0.1
    Y /= Y.sum(axis=0)
    y0 = np.concatenate([rng.uniform(1000.0, 1300.0, (1, n)), Y])
    w = W.Workload("kinetics", W.RHS_KINETICS, W.METHOD_RKC, n, species + 1, np.ascontiguousarray(y0),
                   np.full((1, n), 0.3 * density), 0.0, 2e-7, 1e-6, 1e-10, aux={"mechanism": mech})
    assert_same(w, "rkc")


@pytest.mark.parametrize("bodies", [1, 2, 3, 7, 8, 9, 12, 16])
@pytest.mark.parametrize("method", ["rkck", "rkc"])
def test_nbody_pairs(bodies, method):
    """Each pair formed by one of its two lanes: odd and even rings, 8- and 16-lane teams at their edges."""
    rng = np.random.default_rng(bodies)
    n = 9
    ang = 2 * np.pi * np.arange(bodies) / bodies
    pos = 3.0 * np.stack([np.cos(ang), np.sin(ang)]).reshape(-1, 1) + 0.05 * rng.standard_normal((2 * bodies, n))
    y0 = np.concatenate([pos, 0.5 * rng.standard_normal((2 * bodies, n))])
    w = W.Workload("nbody", W.RHS_NBODY, W.METHOD_RKCK, n, 4 * bodies, np.ascontiguousarray(y0), np.ones((1, n)), 0.0,
                   0.25, 1e-8, 1e-8, aux={"masses": 0.1 * np.arange(1.0, bodies + 1)})
    assert_same(w, method)


@pytest.mark.parametrize("family", ["bruss", "chain"])
@pytest.mark.parametrize("method", ["rkc", "rkck"])
@pytest.mark.parametrize("points,nsys", [(1, 700), (4, 5000), (5, 3001), (8, 3000), (9, 2500), (16, 2500), (17, 1300),
                                         (32, 1301), (33, 5), (33, 700), (64, 650), (40, 7)])
def test_grid_shapes(family, method, points, nsys):
    """Lanes per system by size and batch: both sides of each team width and of the wide kernels."""
    if family == "bruss":
        w = W.bruss(nsys=nsys, n=points, seed=points)
        w.tend = 0.05
    else:
        rng = np.random.default_rng(points)
        w = W.Workload("chain", W.RHS_VDP_CHAIN, W.METHOD_RKCK, nsys, 2 * points,
                       rng.uniform(-2.0, 2.0, (2 * points, nsys)), 10.0 ** rng.uniform(-1.0, 1.0, (1, nsys)), 0.0, 0.2,
                       1e-6, 1e-9)
    assert_same(w, method)


@pytest.mark.parametrize("nsys", [1, 33, 9728, 9729])
@pytest.mark.parametrize("method", ["rkck", "rkc"])
def test_vdp_lanes(nsys, method):
    """Two lanes a system up to a warp per sub-partition (152 SMs: 9728 systems), one past that."""
    w = W.vdp(nsys=nsys, seed=nsys)
    w.tend = 0.5
    assert_same(w, method)


@pytest.mark.parametrize("species,reactions", [(1, 1), (2, 3), (3, 5), (8, 12), (13, 27), (16, 32)])
def test_network_sizes_two_float(species, reactions):
    """Generated two-float networks of odd and even species counts: the packs' unused half, species without a term."""
    import torch
    net = W.make_network(11, species, reactions)
    rng = np.random.default_rng(species)
    n = 65
    y0 = rng.uniform(0.1, 1.0, (species, n))
    w = W.Workload("network", W.RHS_MASSACTION, W.METHOD_RKC, n, species, np.ascontiguousarray(y0 / y0.sum(axis=0)),
                   rng.uniform(1000.0, 2000.0, (1, n)), 0.0, 1e-6, 1e-6, 1e-12, network=net)
    h = B.register_workload(w)
    y = B.integrate("rkc", h, torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda(), w.t0, w.tend, w.rtol,
                    w.atol, precision=B.ODE_PREC_F2_LEAN, sync=True).cpu().numpy()
    B.release(h)
    r = O.integrate(O.model_for(w), W.METHOD_RKC, w.y0, w.params, w.t0, w.tend, w.rtol, w.atol)
    assert (np.abs(y - r.y) / (np.abs(r.y) + w.atol)).max() <= 1e-5  # the two-float form's bar against the FP64 method


@pytest.mark.parametrize("family,nsys", [("mass", 40003), ("mass", 19457), ("bruss", 5003), ("vdp", 100001), ("nbody", 9777)])
def test_parameter_order(family, nsys):
    """Batches that the library takes in parameter order (and n-body, which it does not): same results."""
    w = {"mass": lambda: W.massaction(nsys=nsys, seed=5, tend=2e-7), "bruss": lambda: W.bruss(nsys=nsys, n=32, seed=5),
         "vdp": lambda: W.vdp(nsys=nsys, seed=5), "nbody": lambda: W.pleiades(nsys=nsys, seed=5, tend=0.01)}[family]()
    if family in ("bruss", "vdp"):
        w.tend = 0.05
    assert_same(w, "rkck" if w.method == W.METHOD_RKCK else "rkc")


def test_two_float_order():
    """The two-float network kernel: the order changes no bit."""
    import torch
    w = W.massaction(nsys=70001, seed=6, tend=5e-7)
    h = B.register_workload(w)
    y0, p = torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda()
    out = []
    for cost in (None, torch.ones(w.nsys, dtype=torch.float32, device="cuda")):
        cnt = B.counters_like(w.nsys, "cuda")
        y = B.integrate("rkc", h, y0, p, w.t0, w.tend, w.rtol, w.atol, precision=B.ODE_PREC_F2_LEAN, counters=cnt,
                        cost=cost, mapping=B.ODE_MAP_THREAD, sync=True)
        out.append((y.cpu().numpy(), cnt.n_rhs.cpu().numpy()))
    # 3,000 of the systems as a batch of their own, in their own order
    m = 3000
    y = B.integrate("rkc", h, y0[:, :m].contiguous(), p[:, :m].contiguous(), w.t0, w.tend, w.rtol, w.atol,
                    precision=B.ODE_PREC_F2_LEAN, sync=True).cpu().numpy()
    B.release(h)
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
    np.testing.assert_array_equal(out[0][0][:, :m], y)
