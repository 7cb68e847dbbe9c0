"""The surrogate's training and inference kernels at the edges of their tiles: gradients over batch sizes
around the tile, slot and SM counts, queries around a warp's rows and a full grid, and device arrays
aligned to 4 bytes only."""
import numpy as np
import pytest

from oracle import mlp as M
from test_surrogate import _data, _layer_slices, _theta

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2403_11167_gb300 import lbm as L

    return L


# one sample, a partial and a full smallest tile, one tile per SM of 8 samples and one more, the largest
# tile on every SM and one sample more (some CTAs take two tiles)
@pytest.mark.parametrize("n", [1, 7, 8, 9, 57, 152 * 8, 152 * 8 + 1, 152 * 56, 152 * 56 + 1])
def test_gradient_at_tile_edges(lbm, n):
    """Per tensor within 1e-4 of its largest entry, loss within 1e-5 (the bars of the gradient test),
    and the same bits on a second call."""
    X, Y = _data(max(n, 64), seed=n)
    st = lbm.Surrogate.standardisation(X, Y)
    X, Y = X[:n], Y[:n].copy()
    Y[1::3, 3] = np.nan
    m = lbm.Surrogate(st, seed=1)
    th = _theta(2)
    m.set_params(th)
    loss, g = m.loss_grad(X, Y)
    ref, g_ref = M.loss_grad(th.astype(np.float64), X.astype(np.float64), Y.astype(np.float64), st.astype(np.float64))
    assert abs(loss / ref - 1) < 1e-5
    for sl in _layer_slices():
        assert np.max(np.abs(g[sl] - g_ref[sl])) <= 1e-4 * np.max(np.abs(g_ref[sl])), sl
    again = m.loss_grad(X, Y)
    assert again[0] == loss and np.array_equal(again[1], g)
    m.close()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 152 * 16 + 1, 152 * 12 * 16, 152 * 12 * 16 + 1])
@pytest.mark.parametrize("mode", ["split", "single"])
def test_queries_at_tile_edges(lbm, n, mode):
    """Every standardised output within the first-order rounding bound of its operands (2^-14 split, 2^-8
    single), through device arrays that start 4 bytes off a 16-byte boundary; nothing beyond is written."""
    import torch

    X, _ = _data(max(n, 64), seed=n)
    X = X[:n]
    st = lbm.Surrogate.standardisation(*_data(2000, seed=5))
    m = lbm.Surrogate(st, seed=1)
    th = _theta(5)
    m.set_params(th)
    xin, out = torch.zeros(4 * n + 8, device="cuda"), torch.full((4 * n + 8,), -7.0, device="cuda")
    xin[1:1 + 4 * n] = torch.from_numpy(X.reshape(-1)).cuda()
    torch.cuda.synchronize()
    m.predict_device(xin[1:1 + 4 * n].view(n, 4), out[1:1 + 4 * n].view(n, 4),
                     mode=lbm.LBM_INFER_SPLIT_BF16 if mode == "split" else lbm.LBM_INFER_BF16)
    torch.cuda.synchronize()
    o = out.cpu().numpy()
    assert o[0] == -7.0 and np.all(o[1 + 4 * n:] == -7.0)
    st64 = st.astype(np.float64)
    yn = M.standardise_y(o[1:1 + 4 * n].reshape(n, 4).astype(np.float64), st64)
    ref = M.forward(th.astype(np.float64), M.standardise_x(X.astype(np.float64), st64))[0][-1]
    bound = M.bf16_error_bound(th.astype(np.float64), X.astype(np.float64), st64, u=2.0 ** -14 if mode == "split" else 2.0 ** -8)
    assert np.all(np.abs(yn - ref) <= bound + 1e-5)
    m.close()


@pytest.mark.parametrize("mode", ["split", "single"])
def test_predictions_do_not_depend_on_their_number(lbm, mode):
    """The kernel for few queries (one tile of 16 per CTA to 2432, two above, several rounds to 14592) and
    the one for many: the same bits for the same query."""
    import torch

    sizes = [1, 16, 17, 33, 152 * 16, 152 * 16 + 1, 152 * 32, 152 * 32 + 1, 152 * 64 + 17, 152 * 96, 152 * 96 + 1]
    X, _ = _data(sizes[-1], seed=7)
    m = lbm.Surrogate(lbm.Surrogate.standardisation(X, _data(sizes[-1], seed=7)[1]), seed=1)
    m.set_params(_theta(6))
    x = torch.from_numpy(np.ascontiguousarray(X, dtype=np.float32)).cuda()
    torch.cuda.synchronize()
    got = []
    for n in sizes:
        y = torch.full((n + 1, 4), -7.0, device="cuda")
        torch.cuda.synchronize()
        m.predict_device(x[-n:], y[:n], mode=lbm.LBM_INFER_SPLIT_BF16 if mode == "split" else lbm.LBM_INFER_BF16)
        torch.cuda.synchronize()
        assert bool((y[n:] == -7.0).all())
        got.append(y[:n])
    for y in got[:-1]:
        assert torch.equal(y, got[-1][-len(y):])
    m.close()
