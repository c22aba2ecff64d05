"""One kernel launched from two entry points at once with blocks of different
sizes: 16 bodies' pair planes need the shared-memory opt-in, which belongs to
the kernel, and neither call may lower it under the other's launch."""
import threading

import numpy as np
import pytest

from paper_1611_02274_gb300 import binding as B
from paper_1611_02274_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_blocks_of_two_sizes_at_once():
    import torch
    bodies, n = 16, 64
    rng = np.random.default_rng(0)
    ang = 2 * np.pi * np.arange(bodies) / bodies
    pos = 3.0 * np.stack([np.cos(ang), np.sin(ang)]).reshape(-1, 1) + 0.05 * rng.standard_normal((2 * bodies, n))
    y0 = np.ascontiguousarray(np.concatenate([pos, 0.5 * rng.standard_normal((2 * bodies, n))]))
    w = W.Workload("nbody", W.RHS_NBODY, W.METHOD_RKC, n, 4 * bodies, y0, np.ones((1, n)), 0.0, 1e-3, 1e-6, 1e-6,
                   aux={"masses": 0.1 * np.arange(1.0, bodies + 1)})
    h = B.register_workload(w)
    dy, dp = torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda()
    span = (w.t0, w.tend, w.rtol, w.atol)
    ref = B.integrate("rkc", h, dy, dp, *span, mapping=B.ODE_MAP_THREAD, block_size=256, sync=True).cpu().numpy()
    errors, outs = [], []
    gate = threading.Barrier(2)
    s = torch.cuda.Stream()

    def guarded(f):
        def run():
            gate.wait()
            try:
                for _ in range(400):
                    f()
            except Exception as e:  # noqa: BLE001 -- any error is the finding
                errors.append(e)
        return threading.Thread(target=run)

    y = torch.empty_like(dy)
    threads = [guarded(lambda: B.integrate("rkc", h, dy, dp, *span, y_out=y, mapping=B.ODE_MAP_THREAD, block_size=256,
                                           stream=s.cuda_stream)),
               guarded(lambda: outs.append(B.integrate_noalloc(h, w.y0, w.params, *span, block_size=128)))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    B.release(h)
    assert not errors, errors[0]
    np.testing.assert_array_equal(y.cpu().numpy(), ref)
    for o in outs[::50]:
        np.testing.assert_array_equal(o, ref)
