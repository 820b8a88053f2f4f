"""Field sums of values that lie near 1 in no unit: velocity and area large
together, small together or opposite, so that |u|^2 A or its error terms could
leave the FP32 range although every value lies well within it."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 20000])
@pytest.mark.parametrize("u,a", [(1e13, 1e13), (2e13, 2e13), (1e12, 1e13), (1e13, 1e11), (3e10, 1e12), (1e-10, 1e-12),
                                 (1e-12, 1e-12), (1e-13, 1e-13), (1e-13, 1e-8), (1e-13, 1e-12), (1e13, 1e-13),
                                 (1e-13, 1e13), (1e-5, 1e-13), (1e6, 1e13)])
def test_sums_of_extreme_products(n, u, a):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm as M
    rng = np.random.default_rng(n)
    x = [v.astype(np.float32) for v in (1 + 1e-3 * rng.normal(size=n), u * rng.uniform(0.3, 1.2, n),
                                        -u * rng.uniform(0.3, 1.2, n), a * rng.uniform(0.5, 1.5, n))]
    x[2][::7] = 0
    x[1][::3] *= np.float32(1e-3)  # neighbours on both paths
    d = [torch.from_numpy(v).cuda() for v in x]
    need = M.reduce_scratch_doubles(n)
    scratch, out = (torch.empty(k, dtype=torch.float64, device="cuda") for k in (need, 6))
    M.reduce_fields_device(*[t.data_ptr() for t in d], None, n, scratch.data_ptr(), need, out.data_ptr(),
                           torch.cuda.current_stream().cuda_stream)
    got = out.cpu().numpy()
    r, ux, uy, ar = (v.astype(np.float64) for v in x)
    m2 = ux * ux + uy * uy
    for q, t in enumerate((ar, r * ar, ux * ar, uy * ar, np.sqrt(m2) * ar, m2 * ar)):
        # as FP64 sums: at most four roundings a term, as many for the (at most 20 deep) sums of same-signed terms
        assert abs(got[q] - math.fsum(t)) <= (4 + 20) * 2.0 ** -53 * math.fsum(np.abs(t)), q
