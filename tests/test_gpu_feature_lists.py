"""The features' disk lists where a node's cell lists too few disks, none, or
does not exist, against the oracle."""
import numpy as np
import pytest

from oracle import features as OF
from paper_2312_14789_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm
    return mlbm


@pytest.mark.parametrize("case", ["corner", "ring", "few", "outside"])
def test_features_where_lists_run_short(M, case):
    """Disks in one corner only (most cells list none or one), more disks than
    a block votes on at once, too few for lists, and nodes beyond an open box."""
    rng = np.random.default_rng(5)
    box, sides, L = (0.0, 0.0, 400.0, 300.0), (I.PERIODIC, I.PERIODIC, I.SOLID, I.SOLID), 4.0
    if case == "corner":
        gx, gy = np.meshgrid(np.arange(5), np.arange(4))
        disks = np.stack([20 + 9.0 * gx.ravel(), 20 + 9.0 * gy.ravel(), rng.uniform(2, 4, 20)], 1)
    elif case == "ring":
        gx, gy = np.meshgrid(np.arange(25), np.arange(13))
        disks = np.stack([8 + 16.0 * gx.ravel(), 12 + 22.0 * gy.ravel(), rng.uniform(2, 6, 325)], 1)
    else:
        disks = np.stack([rng.uniform(0, 400, 9), rng.uniform(20, 280, 9), rng.uniform(3, 6, 9)], 1)
    if case == "outside":
        sides = (I.OPEN,) * 4
        gx, gy = np.meshgrid(np.arange(6), np.arange(5))
        disks = np.stack([40 + 60.0 * gx.ravel(), 30 + 55.0 * gy.ravel(), rng.uniform(3, 9, 30)], 1)
    xy = np.stack([rng.uniform(0, 400, 1500), rng.uniform(0, 300, 1500)], 1)
    if case == "outside":
        xy = xy * 1.2 - 30.0
    d = np.min(np.hypot(xy[:, None, 0] - disks[None, :, 0], xy[:, None, 1] - disks[None, :, 1]) - disks[None, :, 2], 1)
    xy = np.ascontiguousarray(xy[d > 0.5])
    X = torch.empty((len(xy), 16), device="cuda")
    M.features_device(xy, box, sides, disks, L, X.data_ptr())
    got, ref = X.cpu().numpy().astype(np.float64), OF.features(xy, box, sides, disks, L)
    # FP32 geometry on coordinates up to 450 gives ~3e-5 in units of L; a choice between two nearly
    # equidistant objects or a grazing ray may fall the other way in a few rows
    assert (np.abs(got - ref).max(1) > 1e-4).mean() <= 0.01
