"""What a small plain FP64 batch launches does not depend on the batches
before it: the mapping timed for a large batch is for large batches."""
import numpy as np
import pytest

from paper_1611_02274_gb300 import binding as B
from paper_1611_02274_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_small_batches_keep_the_default():
    import torch
    prec = B.ODE_PREC_FP64
    small, large = W.vdp(100, seed=1), W.vdp(40000, seed=2)
    small.tend = large.tend = 0.5
    h = B.register_workload(small)

    def run(w):
        y = B.integrate("rkck", h, torch.from_numpy(w.y0).cuda(), torch.from_numpy(w.params).cuda(), w.t0, w.tend,
                        w.rtol, w.atol, precision=prec, sync=True).cpu().numpy()
        return y, B.last_launch()

    y, info = run(small)
    want = {"ordered": False, "lanes": 2, "block": 32, "mapping": B.ODE_MAP_THREAD}
    assert info == want
    _, tuned = run(large)
    m, b, is_tuned = B.mapping_info(h, "rkck", prec)
    assert is_tuned and (tuned["mapping"], tuned["block"]) == (m, b)
    y2, info2 = run(small)
    B.release(h)
    assert info2 == want
    np.testing.assert_array_equal(y2, y)
