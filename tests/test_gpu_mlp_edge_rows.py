"""No row of a minibatch is lost where the gradient kernel's tiles, rounds and block
ranges end: the targets equal the network's own outputs except on a few rows at
those edges, so that loss and gradient come from these rows alone and a lost one
changes both by about its share."""
import numpy as np
import pytest

from oracle import mlp as OM

torch = pytest.importorskip("torch")

TILE, ROUND, BLOCKS = 16, 128, 152  # rows of a tile and of a block's round, most blocks


def _edge_rows(n):
    """First and last row of the set, of a block's range, of its last tile, and of its rounds."""
    tiles, blocks = -(-n // TILE), min(-(-n // ROUND), BLOCKS)
    start = [tiles * b // blocks for b in range(blocks + 1)]
    rows = {0, n - 1, (tiles - 1) * TILE}
    for b in {0, blocks - 1, *[b for b in range(blocks) if start[b + 1] - start[b] > ROUND // TILE][:1]}:
        a, e = start[b] * TILE, min(n, start[b + 1] * TILE)
        rows |= {a, e - 1, max(a, e - TILE), min(e - 1, a + ROUND - 1), min(e - 1, a + ROUND)}
    return np.array(sorted(rows))


def _net(no):
    rng = np.random.default_rng(no)
    parts = []
    for a, b in ((16, 64), (64, 64), (64, 64), (64, no)):
        parts += [rng.normal(0, (2 / a) ** 0.5, a * b), rng.normal(0, 0.1, b)]
    return np.concatenate(parts).astype(np.float32)


def _rows_gradient(flat, x, t, no):
    """Sum over rows of the squared error's gradient."""
    return len(x) * OM.pack(OM.gradients(OM.unpack(flat.astype(np.float64), no), x, t, bf16_round=True))


SIZES = [1, 17, 129, 143, 2049, 19456, 19457, 20000, 39001]
TOL = 0.04  # of the gradient's norm: BF16 roundings that fall the other way; a lost row changes it by more, see below


@pytest.mark.gpu
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("no", [1, 2, 3])
def test_every_edge_row_counts(n, no):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm as M
    flat, rows = _net(no), _edge_rows(n)
    net = M.Mlp(3, no)
    net.set_params(flat)
    x = np.random.default_rng(n).normal(size=(n, 16)).astype(np.float32)
    X, T = torch.from_numpy(x).cuda(), torch.empty((n, no), device="cuda")
    net.forward(X.data_ptr(), n, T.data_ptr())
    torch.cuda.synchronize()
    y = T.cpu().numpy()
    T[rows] += 1.0
    t = T.cpu().numpy()
    G = torch.empty(net.param_count(), device="cuda")
    loss = net.gradients(X.data_ptr(), T.data_ptr(), n, G.data_ptr())
    # every edge row adds the square of the FP32 errors it was given, every other row nothing above FP32 round-off
    want = ((y.astype(np.float64) - t.astype(np.float64))[rows].astype(np.float32).astype(np.float64) ** 2).sum()
    assert abs(loss * n - want) <= 1e-5 * want
    g = G.cpu().numpy().astype(np.float64) * n
    ref = _rows_gradient(flat, x[rows].astype(np.float64), t[rows].astype(np.float64), no)
    assert np.linalg.norm(g - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("no", [1, 2, 3])
def test_a_lost_row_would_show(n, no):
    """The same sums in the oracle without one of the rows are further off than the tolerance."""
    flat, rows = _net(no), _edge_rows(n)
    x = np.random.default_rng(n).normal(size=(n, 16)).astype(np.float32)[rows].astype(np.float64)
    y, _ = OM.forward(OM.unpack(flat.astype(np.float64), no), x, bf16_round=True)
    t = y + 1.0
    whole = _rows_gradient(flat, x, t, no)
    for k in range(len(rows)):
        keep = np.arange(len(rows)) != k
        rest = _rows_gradient(flat, x[keep], t[keep], no) if keep.any() else 0 * whole
        assert np.linalg.norm(whole - rest) > 1.5 * TOL * np.linalg.norm(whole), (n, no, rows[k])
