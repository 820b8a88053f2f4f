"""The field sums formed on the FP32 pipe, at sizes around their blocks and for
values that leave its range."""
import math

import numpy as np
import pytest

from paper_2312_14789_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm
    return mlbm


def _sums(M, rho, ux, uy, area, mask):
    n = len(rho)
    d = [torch.from_numpy(a).cuda() for a in (rho, ux, uy, area)]
    m = None if mask is None else torch.from_numpy(mask).cuda()
    need = M.reduce_scratch_doubles(n)
    scratch, out = torch.empty(need, dtype=torch.float64, device="cuda"), torch.empty(6, dtype=torch.float64, device="cuda")
    M.reduce_fields_device(*[t.data_ptr() for t in d], None if m is None else m.data_ptr(), n, scratch.data_ptr(), need,
                           out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    return out.cpu().numpy()


def _terms(rho, ux, uy, area, mask):
    keep = np.ones(len(rho), bool) if mask is None else mask != 0
    r, u, v, a = (x[keep].astype(np.float64) for x in (rho, ux, uy, area))
    with np.errstate(all="ignore"):
        m2 = u * u + v * v
        return [a, r * a, u * a, v * a, np.sqrt(m2) * a, m2 * a]


@pytest.mark.parametrize("n", [1, 2, 1023, 1025, 155648, 155649, 700001])
@pytest.mark.parametrize("values", ["flow", "scales", "tiny", "huge", "still"])
def test_sums_against_exactly_rounded(M, n, values):
    rng = np.random.default_rng(n)
    rho, area = 1 + 1e-3 * rng.normal(size=n), rng.uniform(0.2, 1.5, n)
    ux, uy = 1e-2 * rng.normal(size=n) + 3e-3, 1e-2 * rng.normal(size=n)
    if values == "scales":  # from far below to far above the FP32 pipe's range, within one sum
        ux, uy = ux * 10.0 ** rng.uniform(-25, 17, n), uy * 10.0 ** rng.uniform(-25, 17, n)
    elif values == "tiny":
        ux, uy = ux * 1e-28, uy * 1e-30
    elif values == "huge":
        ux, area = ux * 1e20, area * 1e16
    elif values == "still":
        ux, uy = ux * 0, np.where(rng.random(n) < 0.5, 0, uy)
    a = [x.astype(np.float32) for x in (rho, ux, uy, area)]
    for mask in (None, (rng.random(n) < 0.8).astype(np.uint8)):
        got = _sums(M, *a, mask)
        for q, t in enumerate(_terms(*a, mask)):
            # a term carries at most four roundings of 2^-53 in either form, a sum of sums the same again
            assert abs(got[q] - math.fsum(t)) <= 1e-15 * math.fsum(np.abs(t)), q


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_sums_pass_infinities_on(M, bad):
    n = 3000
    rng = np.random.default_rng(1)
    a = [x.astype(np.float32) for x in (1 + rng.random(n), rng.random(n), rng.random(n), 1 + rng.random(n))]
    a[1][1234] = bad
    got, ref = _sums(M, *a, None), np.array([np.sum(t) for t in _terms(*a, None)])
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    assert np.allclose(got[[0, 1, 3]], ref[[0, 1, 3]], rtol=1e-12)


def test_macroscopics_is_the_fields_apart(M):
    w = I.porous(seed=3, n_target=2000)
    st = M.build_stencils_for(w, K=16, s=1.0)
    for p in (M.Params(M.MODEL_BGK, 0.8, 0.0, 1e-5, 2e-6), M.Params(M.MODEL_TAU1, 1.0, 0.0, 1e-5, 0.0)):
        ctx = M.init(st, p)
        M.step(ctx, 9)
        ru = M.get_fields(ctx)
        rho, u = M.macroscopics(ctx)
        assert np.array_equal(rho, ru[:, 0]) and np.array_equal(u, ru[:, 1:])

