"""The network's gradient and training kernels at the row counts where their
16-row tiles, 128-row rounds and per-block ranges end, and the weight image
after parameters change, against the oracle's network, which rounds to BF16
where the kernels do."""
import numpy as np
import pytest

from oracle import mlp as OM

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup(n, no, seed):
    from paper_2312_14789_gb300 import mlbm as M
    rng = np.random.default_rng(seed)
    parts = []
    for a, b in ((16, 64), (64, 64), (64, 64), (64, no)):
        parts += [rng.normal(0, (2 / a) ** 0.5, a * b), rng.normal(0, 0.1, b)]
    flat = np.concatenate(parts).astype(np.float32)
    net = M.Mlp(3, no)
    net.set_params(flat)
    X = torch.from_numpy(rng.normal(size=(n, 16)).astype(np.float32)).cuda()
    T = torch.from_numpy(rng.normal(size=(n, no)).astype(np.float32)).cuda()
    return net, flat, X, T


@pytest.mark.parametrize("n", [1, 15, 16, 17, 127, 128, 129, 143, 19456, 19457, 20000])
@pytest.mark.parametrize("no", [1, 2, 3])
def test_gradients_at_the_edges_of_a_round(n, no):
    net, flat, X, T = _setup(n, no, 10 * n + no)
    G = torch.empty(net.param_count(), device="cuda")
    loss = net.gradients(X.data_ptr(), T.data_ptr(), n, G.data_ptr())
    p = OM.unpack(flat.astype(np.float64), no)
    x, t = X.cpu().numpy().astype(np.float64), T.cpu().numpy().astype(np.float64)
    y, _ = OM.forward(p, x, bf16_round=True)
    g = OM.pack(OM.gradients(p, x, t, bf16_round=True))
    ref = float(((y - t) ** 2).sum() / n)
    # far above what another order of FP32 sums does through the BF16 roundings, far below a lost tile, row or column
    assert abs(loss - ref) < 0.03 * ref
    assert np.linalg.norm(G.cpu().numpy() - g) < 0.05 * np.linalg.norm(g)
    Y = torch.empty((n, no), device="cuda")
    net.forward(X.data_ptr(), n, Y.data_ptr())
    torch.cuda.synchronize()
    assert np.linalg.norm(Y.cpu().numpy() - y) < 0.03 * np.linalg.norm(y)


def test_training_moves_image_and_parameters_together():
    """After training, inference uses the trained parameters (a network loaded
    with them predicts the same bits), and a repeated run gives the same bits."""
    from paper_2312_14789_gb300 import mlbm as M
    net, flat, X, T = _setup(5000, 3, 4)
    net.train(X.data_ptr(), T.data_ptr(), 5000, 1000, 7, 1e-3, 99)
    p = net.get_params()
    assert np.abs(p - flat).max() > 1e-4
    again, _, _, _ = _setup(5000, 3, 4)
    again.train(X.data_ptr(), T.data_ptr(), 5000, 1000, 7, 1e-3, 99)
    assert np.array_equal(again.get_params(), p)
    other = M.Mlp(8, 3)
    other.set_params(p)
    a, b = torch.empty((5000, 3), device="cuda"), torch.empty((5000, 3), device="cuda")
    net.forward(X.data_ptr(), 5000, a.data_ptr())
    other.forward(X.data_ptr(), 5000, b.data_ptr())
    torch.cuda.synchronize()
    assert torch.equal(a, b)
