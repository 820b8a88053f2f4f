"""The lattice wall force, summed from the device's own state in 64 bits over the
links that come from a solid cell: the list of wall links holds each of them once,
at periodic seams and open sides, in boxes one cell wide too."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
EY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
W32 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, np.float32)  # as the device subtracts them
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]


def _links(cell, periodic, k):
    """Fluid cells whose population k arrives from a solid cell (inside the box, or across a periodic side)."""
    link = (cell == 0) & np.roll(cell == 1, (EY[k], EX[k]), (0, 1))
    if EX[k] and not periodic[0]:
        link[:, 0 if EX[k] > 0 else -1] = False
    if EY[k] and not periodic[1]:
        link[0 if EY[k] > 0 else -1] = False
    return link


@pytest.mark.parametrize("nx,ny", [(64, 4), (65, 5), (1, 9), (9, 1), (2, 2), (130, 33), (257, 40)])
@pytest.mark.parametrize("periodic", [(True, True), (True, False), (False, True), (False, False)])
def test_force_of_the_listed_links(nx, ny, periodic):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm as M
    rng = np.random.default_rng(nx * 1000 + ny)
    cell = np.zeros((ny, nx), np.uint8)
    cell[rng.random((ny, nx)) < 0.15] = 1
    cell[rng.random((ny, nx)) < 0.05] = 2
    cell.flat[0], cell.flat[-1] = 1, 0  # a solid corner, and a fluid one that sees it across the seams
    eqv = np.stack([1 + 0.01 * rng.random((ny, nx)), 0.02 * rng.random((ny, nx)), -0.02 * rng.random((ny, nx))], -1)
    f = W32 * (1 + 0.05 * rng.normal(size=(ny, nx, 9)))
    L = M.Lattice(cell, M.Params(M.MODEL_BGK, 0.8, 0.0, 0.0, 0.0), periodic=periodic, eq_values=eqv)
    L.set_populations(f)
    for steps in (0, 17):
        L.step(steps)
        g = L.get_populations().reshape(ny, nx, 9) - W32.astype(np.float64)
        terms = [(2 * g[..., OPP[k]][_links(cell, periodic, k)], k) for k in range(1, 9)]
        got = L.force()
        for axis, e in ((0, EX), (1, EY)):
            v = np.concatenate([t * e[OPP[k]] for t, k in terms])
            # a population read back carries a rounding of 2^-54 (it was added to a weight), the sums as many
            # roundings of their partial sums; a link left out is worth its population, typically 1e-3
            assert abs(got[axis] - math.fsum(v)) <= 1e-13 * (len(v) + 1), (steps, axis)
