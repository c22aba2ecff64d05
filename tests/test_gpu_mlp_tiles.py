"""The training kernels' tiles against the FP64 reference network: row counts
around a tile of 32 and past one tile per resident block, and input counts
around the padded quarters of the first layer's gradient."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_1611_02274_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n_in", [(1, 14), (31, 1), (32, 4), (33, 16), (700, 17), (20011, 14), (65, 33)])
def test_gradient_tiles(rows, n_in):
    import torch
    rng = np.random.default_rng(rows + n_in)
    net = B.MLP(n_in, seed=n_in)
    norm = np.zeros(M.NORM_SIZE, dtype=np.float32)
    norm[:n_in] = rng.normal(size=n_in)
    norm[33:33 + n_in] = rng.uniform(0.5, 2.0, size=n_in)
    norm[66:66 + n_in], norm[99:99 + n_in] = -1e30, 1e30
    norm[132:135], norm[135:138] = rng.normal(size=3), rng.uniform(0.5, 2.0, size=3)
    net.set_params(norm=norm)
    X = rng.normal(size=(rows, n_in)).astype(np.float32)
    Y = rng.normal(size=(rows, 3)).astype(np.float32)
    Y[::5, 2] = np.nan  # a missing target adds nothing
    params, _ = net.get_params()
    g, loss = net.gradient(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda())
    ref_loss, ref = M.loss_and_grad(M.bf16_round(params), norm, X, Y)
    net.release()
    g = g.cpu().numpy()
    # every term carries the fast exponential's ~1e-6 and FP32 sums a few ulp
    # more; where terms cancel, that is relative to the largest gradient
    assert loss == pytest.approx(ref_loss, rel=1e-4)
    np.testing.assert_allclose(g, ref, rtol=1e-3, atol=1e-5 * np.abs(ref).max())


def test_training_is_reproducible():
    """The blocks' sums are taken in a fixed order: two runs agree bit for bit."""
    import torch
    rng = np.random.default_rng(4)
    X = torch.from_numpy(rng.normal(size=(5000, 6)).astype(np.float32)).cuda()
    Y = torch.from_numpy(rng.normal(size=(5000, 3)).astype(np.float32)).cuda()
    out = []
    for _ in range(2):
        net = B.MLP(6, seed=1)
        net.fit_normalization(X, Y)
        hist = net.train(X, Y, epochs=2, batch=1000, seed=3)
        out.append((net.get_params()[0], hist))
        net.release()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
