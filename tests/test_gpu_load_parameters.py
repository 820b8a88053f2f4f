"""A checkpoint brings its parameters along: after a load every later step, also
one replayed from a graph that was captured before, and every time scale taken
from the parameters are those of the file."""
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


@pytest.mark.parametrize("n", [1200, 9000])  # steps by one cluster launch, and by replayed graphs
@pytest.mark.parametrize("batch_of_one", [False, True])
def test_steps_after_a_load_use_the_loaded_parameters(M, tmp_path, n, batch_of_one):
    w = I.porous(seed=5, n_target=n)
    st = M.build_stencils_for(w, K=16, s=0.5)
    old, new = M.Params(M.MODEL_BGK, 0.8, 0.0, 1e-6, 0.0), M.Params(M.MODEL_BGK, 0.65, 1.3, 4e-5, 1e-5)

    def make(p):
        return M.batch_init([st], [p]) if batch_of_one else M.init(st, p)

    src, ctx, ref = make(new), make(old), make(new)
    M.step(src, 5)
    path = str(tmp_path / "state")
    M.save(src, path)
    M.step(ctx, 33)  # graphs of both buffers
    M.step(ctx, 32)
    M.load(ctx, path)
    M.step(ref, 5)
    for c in (ctx, ref):
        M.step(c, 48)
    a, b = M.get_populations(ctx), M.get_populations(ref)
    assert np.isfinite(b).all() and np.array_equal(a, b)


def test_steady_criterion_after_a_load_uses_the_loaded_time_scale(M, tmp_path):
    """Without a time step of the caller's the mean-velocity criterion takes it from tau."""
    w = I.porous(seed=5, n_target=3000)
    st = M.build_stencils_for(w, K=16, s=1.0)
    old, new = M.Params(M.MODEL_BGK, 0.51, 0.0, 1e-6, 0.0), M.Params(M.MODEL_BGK, 1.0, 0.0, 1e-6, 0.0)
    src, ctx = M.init(st, new), M.init(st, old)
    path = str(tmp_path / "state")
    M.save(src, path)
    M.load(ctx, path)
    taken = [M.run_to_steady_mean(c, threshold=2.0, dn=50, check=50, max_steps=20000) for c in (src, ctx)]
    assert taken[0] == taken[1] and 100 < taken[0] < 20000
