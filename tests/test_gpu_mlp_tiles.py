"""Surrogate kernels at the edges of their row tiles, against the oracle.

The forward pass takes 16, 32 or 64 rows per CTA and the training pass 16 or
32, by the number of 16-row tiles against the SMs of the device; the weight
gradients sum chunks of 512 rows.  Bounds as in the oracle
comparison of the other surrogate tests: equal bf16 roundings, so only the
FP32 summation order and tipped bf16 decisions differ (2e-3 of the output
scale, 2e-2 of a block's largest gradient).
"""
import numpy as np
import pytest

from oracle import mlp_oracle as M

pytestmark = pytest.mark.gpu


def _rows():
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
    # one row, tile and chunk edges, one and two tiles per SM, and beyond
    return [1, 15, 17, 512, 513, 16 * sms, 16 * sms + 1, 32 * sms, 32 * sms + 33]


def _net(n):
    from paper_0807_0602_gb300.build import build
    build()
    from paper_0807_0602_gb300 import surrogate
    th = surrogate.init_params(7)
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, 6)).astype(np.float32)
    T = rng.normal(size=(n, 3)).astype(np.float32)
    return surrogate.Network(max_batch=n, params=th), th.astype(np.float64), X, T


@pytest.mark.parametrize("case", range(9))
def test_forward_and_gradients_at_tile_edges(case):
    n = _rows()[case]
    net, th, X, T = _net(n)
    y = net.forward(X).cpu().numpy()
    yb, _ = M.forward(th, X.astype(np.float64), bf16=True)
    assert np.max(np.abs(y - yb)) <= 2e-3 * max(np.abs(yb).max(), 1e-3)
    g, loss = net.gradients(X, T)
    g = g.cpu().numpy()
    lb, gb = M.backward(th, X.astype(np.float64), T.astype(np.float64), bf16=True)
    assert abs(float(loss) - lb) <= 1e-3 * lb
    off = 0
    for a, b in ((6, 128), (128, 128), (128, 128), (128, 3)):
        for size in (a * b, b):
            gk, bk = g[off:off + size], gb[off:off + size]
            off += size
            assert np.max(np.abs(gk - bk)) <= 2e-2 * np.max(np.abs(bk)), (n, a, b, size)
    net.close()


@pytest.mark.parametrize("n", [1, 16, 65, 512])
def test_gathered_minibatches_equal_single_steps(n):
    """train_steps on row numbers = train_step on the gathered rows, bit for bit
    (rows repeat and are out of order; n = 512 fills one chunk of the sums)."""
    import torch
    from paper_0807_0602_gb300 import surrogate
    rows = 700
    a, th, X, T = _net(rows)
    b = surrogate.Network(max_batch=rows, params=th.astype(np.float32))
    idx = np.random.default_rng(3).integers(0, rows, size=(5, n))
    la = a.train_steps(X, T, idx, 1e-3).cpu().numpy()
    lb = torch.cat([b.train_step(X[i], T[i], 1e-3) for i in idx]).cpu().numpy()
    assert np.array_equal(la, lb) and np.array_equal(a.params, b.params) and a.steps == b.steps == 5
    a.close()
    b.close()


@pytest.mark.parametrize("where", ["numpy", "cuda"])
def test_row_numbers_out_of_range_are_refused(where):
    """(The kernel reads row 0 for them: nothing is trained on a wrong row.)"""
    import torch
    rows = 40
    net, th, X, T = _net(rows)
    for bad in (-1, rows, 1 << 40):
        idx = np.arange(16).reshape(2, 8)
        idx[1, 3] = bad
        with pytest.raises(IndexError):
            net.train_steps(X, T, idx if where == "numpy" else torch.as_tensor(idx, device="cuda"), 1e-3)
    assert net.steps == 0 and np.array_equal(net.params, th.astype(np.float32))
    assert net.train_steps(X, T, np.array([[0, rows - 1]]), 1e-3).shape == (1,)
    net.close()
