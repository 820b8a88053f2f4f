"""The bounded wait of a cluster run: when one block's records never arrive, the
other blocks are not left waiting for it, the launch ends, the call that follows
reports the wait, and the context goes on from a clean state.  Nothing faults: the
block steps nothing, and meets the others at every barrier."""
import numpy as np
import pytest

from paper_2312_14789_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,steps", [(25, 8), (600, 9), (2000, 40)])  # one block, and sixteen of two and four tiles
@pytest.mark.parametrize("K", [12, 16])
def test_withheld_records_time_out_and_the_context_recovers(nodes, steps, K):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm as M
    w = I.poiseuille_channel(nodes // 5, 5, 0.2, seed=1)
    st = M.build_stencils_for(w, K=K, s=1.0, bb_mode=M.BB_INTERPOLATED)
    ref, ctx = (M.init(st, M.Params(M.MODEL_BGK, 0.8, 0.0, 1e-5, 0.0)) for _ in range(2))
    M.set_wait_limit(ctx, 1e-3)
    ru = np.stack([1 + 1e-3 * np.sin(w.xy[:, 0]), 0.01 * np.cos(w.xy[:, 1]), np.zeros(w.n)], 1)
    for c in (ref, ctx):
        M.set_fields(c, ru)
    M.test_withhold_copy(ctx)
    M.step(ctx, steps)
    with pytest.raises(M.MlbmError) as e:
        M.get_fields(ctx)
    assert e.value.status == 6, str(e.value)
    M.set_fields(ctx, ru)
    for c in (ref, ctx):
        M.step(c, steps)
    assert np.array_equal(M.get_populations(ctx), M.get_populations(ref))
