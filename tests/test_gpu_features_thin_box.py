"""Geometry features of a box far longer than wide with many disks: the disk lists
stay within their bound (one cell across, cells of a quarter of the reach along
would list 10^5 disks for each of 9 10^5 cells, more than the device holds)."""
import numpy as np
import pytest

from oracle import features as OF
from paper_2312_14789_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("along", [0, 1])
def test_features_of_a_thin_box_with_many_disks(along):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm as M
    rng = np.random.default_rng(3)
    nd, long, wide = 100_000, 1e7, 1e-3
    disks = np.stack([100.0 * np.arange(nd), np.full(nd, 5e-4), rng.uniform(5e-5, 2e-4, nd)], 1)
    xy = np.stack([100.0 * (np.arange(24) % 3) + rng.uniform(2.5e-4, 6e-4, 24), rng.uniform(0, 1e-3, 24)], 1)
    box, sides = (-50.0, 0.0, long - 50.0, wide), (I.OPEN, I.OPEN, I.SOLID, I.SOLID)
    if along:  # the long way up
        disks, xy = disks[:, [1, 0, 2]], xy[:, ::-1]
        box, sides = (0.0, -50.0, wide, long - 50.0), (I.SOLID, I.SOLID, I.OPEN, I.OPEN)
    disks, xy = np.ascontiguousarray(disks), np.ascontiguousarray(xy)
    X = torch.empty((len(xy), 16), device="cuda")
    M.features_device(xy, box, sides, disks, 1e-4, X.data_ptr())
    # only the first disks are within 4 L of a node; the porosity of the box (feature 14) counts them all
    got, ref = X.cpu().numpy().astype(np.float64), OF.features(xy, box, sides, disks[:6], 1e-4)
    ref[:, 14] = 1 - np.pi * np.sum(disks[:, 2] ** 2) / (long * wide)
    # FP32 geometry on coordinates up to 10 L; positions 250 from the corner as 48-bit pairs are exact to 10^-8 L
    err = np.abs(got - ref).max(1)
    assert (err > 1e-4).sum() <= 1 and np.isfinite(got).all()
