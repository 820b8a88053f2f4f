"""The geometry features of a box far from the origin: with coordinates that a
double holds exactly on both sides of the shift, every displacement is the same
number, and so is every feature."""
import numpy as np
import pytest

from paper_2312_14789_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PERIODIC_SOLID = (I.PERIODIC, I.PERIODIC, I.SOLID, I.SOLID)


@pytest.mark.parametrize("shift", [(2.0 ** 30, -2.0 ** 29), (-2.0 ** 24, 2.0 ** 30)])
@pytest.mark.parametrize("sides", [PERIODIC_SOLID, (I.PERIODIC,) * 4, (I.OPEN,) * 4])
@pytest.mark.parametrize("n_disks", [9, 60])  # looked at one by one, and listed per cell
def test_features_do_not_depend_on_the_origin(shift, sides, n_disks):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm as M
    rng = np.random.default_rng(n_disks)

    def grid(v):  # multiples of 2^-22: 52 bits at the far end
        return np.round(v * 2.0 ** 22) / 2.0 ** 22

    disks = np.stack([grid(rng.uniform(0, 384, n_disks)), grid(rng.uniform(8, 300, n_disks)),
                      rng.uniform(2, 5, n_disks)], 1)
    xy = np.ascontiguousarray(np.stack([grid(rng.uniform(0, 384, 3000)), grid(rng.uniform(0, 320, 3000))], 1))
    out = []
    for ox, oy in ((0.0, 0.0), shift):
        d = disks + np.array([ox, oy, 0.0])
        p = xy + np.array([ox, oy])
        X = torch.empty((len(xy), 16), device="cuda")
        M.features_device(p, (ox, oy, ox + 384.0, oy + 320.0), sides, d, 4.0, X.data_ptr())
        out.append(X)
    assert torch.equal(out[0], out[1])
