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


@pytest.mark.parametrize("n", [255, 257, 511, 512, 513])
def test_sums_of_one_or_two_nodes_a_thread(n):
    """The FP64 form that short arrays take, and the first length that does not, on ordinary values; the
    sums of a context that short take the same form."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import inputs as I
    from paper_2312_14789_gb300 import mlbm as M
    rng = np.random.default_rng(n)
    x = [v.astype(np.float32) for v in (1 + 1e-3 * rng.normal(size=n), 1e-2 * rng.normal(size=n),
                                        1e-2 * rng.normal(size=n), rng.uniform(0.5, 1.5, n))]
    mask = (rng.random(n) < 0.7).astype(np.uint8)
    d = [torch.from_numpy(v).cuda() for v in x + [mask]]
    need = M.reduce_scratch_doubles(n)
    scratch, out = (torch.empty(k, dtype=torch.float64, device="cuda") for k in (need, 6))
    M.reduce_fields_device(*[t.data_ptr() for t in d], n, scratch.data_ptr(), need, out.data_ptr(),
                           torch.cuda.current_stream().cuda_stream)
    got = out.cpu().numpy()
    r, ux, uy, ar = (v.astype(np.float64)[mask != 0] for v in x)
    for q, t in enumerate((ar, r * ar, ux * ar, uy * ar, np.hypot(ux, uy) * ar, (ux * ux + uy * uy) * ar)):
        assert abs(got[q] - math.fsum(t)) <= (4 + 20) * 2.0 ** -53 * math.fsum(np.abs(t)), q
    # a channel of 512 nodes, and of 533: superficial velocity from its own sums
    w = I.poiseuille_channel(32 if n <= 512 else 41, 16 if n <= 512 else 13, 0.2, seed=1)
    ctx = M.init(M.build_stencils_for(w, K=12, s=1.0), M.Params(M.MODEL_BGK, 0.8, 0.0, 1e-4, 0.0))
    M.step(ctx, 20)
    ru = M.get_fields(ctx)
    assert not (w.node_class == M.NODE_EQ).any()
    ref = math.fsum(ru[:, 1] * w.area.astype(np.float32).astype(np.float64))
    box = (w.box[2] - w.box[0]) * (w.box[3] - w.box[1])
    assert abs(M.permeability(ctx)["u_superficial"] * box - ref) <= 1e-12 * abs(ref)
