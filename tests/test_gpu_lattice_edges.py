"""The lattice step where its blocks, wrap-arounds and graph replays can go
wrong: sizes around the 64 x 4 blocks, one-cell-wide boxes, mixed periodic
sides with solid and equilibrium cells, and step counts around a captured
graph, against a plain numpy step in 64 bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
EY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]


def _feq(rho, ux, uy):
    eu = ux[..., None] * EX + uy[..., None] * EY
    return W * rho[..., None] * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy)[..., None])


def _step(f, cell, eqv, periodic, tau):
    ny, nx = cell.shape
    g = np.empty_like(f)
    for k in range(9):
        src = np.roll(f[..., k], (EY[k], EX[k]), (0, 1))
        bounce = np.roll(cell == 1, (EY[k], EX[k]), (0, 1))
        if EX[k] and not periodic[0]:
            bounce[:, 0 if EX[k] > 0 else -1] = True
        if EY[k] and not periodic[1]:
            bounce[0 if EY[k] > 0 else -1] = True
        g[..., k] = np.where(bounce, f[..., OPP[k]], src)
    rho = g.sum(-1)
    ux, uy = (g @ EX) / rho, (g @ EY) / rho
    out = g - (g - _feq(rho, ux, uy)) / tau
    out = np.where((cell == 2)[..., None], _feq(eqv[..., 0], eqv[..., 1], eqv[..., 2]), out)
    return np.where((cell == 1)[..., None], f, out)


@pytest.mark.parametrize("nx,ny", [(64, 4), (65, 5), (63, 3), (1, 9), (9, 1), (130, 33)])
@pytest.mark.parametrize("periodic", [(True, True), (True, False), (False, False)])
def test_lattice_edges(nx, ny, periodic):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm as M
    rng = np.random.default_rng(nx * 1000 + ny)
    cell = np.zeros((ny, nx), np.uint8)
    if nx * ny > 64:
        cell[rng.random((ny, nx)) < 0.1] = 1
        cell[rng.random((ny, nx)) < 0.05] = 2
    eqv = np.stack([1 + 0.01 * rng.random((ny, nx)), 0.02 * rng.random((ny, nx)), -0.02 * rng.random((ny, nx))], -1)
    f = _feq(1 + 0.01 * rng.random((ny, nx)), 0.03 * rng.random((ny, nx)), 0.03 * rng.random((ny, nx)))
    f[cell == 1] = W  # solid cells are never written: both buffers hold the rest state
    L = M.Lattice(cell, M.Params(M.MODEL_BGK, 0.8, 0.0, 0.0, 0.0), periodic=periodic, eq_values=eqv)
    L.set_populations(f)
    for steps in (1, 16, 19, 34):
        L.step(steps)
        for _ in range(steps):
            f = _step(f, cell, eqv, periodic, 0.8)
        # round-off of ~40 FP32 operations on deviations below 0.05 per step, not amplified by the stable collision
        assert np.abs(L.get_populations().reshape(ny, nx, 9) - f).max() < 70 * 40 * 2.0 ** -24 * 0.05
    fx = fy = 0.0
    for k in range(1, 9):
        link = (cell == 0) & np.roll(cell == 1, (EY[k], EX[k]), (0, 1))
        if EX[k] and not periodic[0]:
            link[:, 0 if EX[k] > 0 else -1] = False
        if EY[k] and not periodic[1]:
            link[0 if EY[k] > 0 else -1] = False
        v = 2 * (f[..., OPP[k]] - W[k])[link].sum()
        fx += v * EX[OPP[k]]
        fy += v * EY[OPP[k]]
    got = L.force()
    links = 8 * int((cell == 0).sum())
    assert max(abs(got[0] - fx), abs(got[1] - fy)) < 2 * links * 70 * 40 * 2.0 ** -24 * 0.05
