"""Which kernel steps an RBF-FD context follows from its size and kernel variant
alone, not from the calls that came before; the autotuner times and keeps the
kernel that the chosen variant then runs."""
import numpy as np
import pytest

from paper_2312_14789_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RECORDS = "step_rbf_tiles"


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_14789_gb300 import mlbm
    _profile(lambda: torch.zeros(9, device="cuda").add_(1))  # the first profile of a process may miss its kernels
    if "add" not in _profile(lambda: torch.zeros(9, device="cuda").add_(1)):
        pytest.skip("the profiler records no kernels here")
    return mlbm


def _profile(call):
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return " ".join(e.key for e in prof.key_averages())


def _kernels(call):
    names = _profile(call)
    assert "step" in names
    return names


def _context(M):
    w = I.poiseuille_channel(60, 40, 0.2, seed=4)
    st = M.build_stencils_for(w, K=24, s=0.5, bb_mode=1, interp=M.INTERP_RBF)
    return M.init(st, M.Params(M.MODEL_BGK, 0.8, 1.1, 1e-5, 0.0))


def test_records_step_under_28_and_29_only(M):
    ctx = _context(M)
    for variant in (27, 28, 27, 1, 29, 25):
        M.set_kernel_variant(ctx, variant)
        assert (RECORDS in _kernels(lambda: M.step(ctx, 3))) == (variant in (28, 29)), variant


def test_autotune_times_the_records(M):
    ctx, ref = _context(M), _context(M)
    assert RECORDS in _kernels(lambda: M.autotune(ctx, 4))
    chosen = M.kernel_variant(ctx)
    assert (RECORDS in _kernels(lambda: M.step(ctx, 3))) == (chosen in (28, 29)), chosen
    M.step(ref, 3)
    assert np.array_equal(M.get_populations(ctx), M.get_populations(ref))


@pytest.mark.parametrize("nx,ny,large", [(160, 150, False), (190, 145, True), (300, 157, True)])
def test_large_sets_step_from_records_by_default(M, nx, ny, large):
    """Plain rows of 55, 63 and 109 MB: records from 60 MB on."""
    w = I.poiseuille_channel(nx, ny, 0.2, seed=4)
    st = M.build_stencils_for(w, K=64, s=0.5, bb_mode=1, interp=M.INTERP_RBF_POINTS, n_l=25)
    ctx, ref = (M.init(st, M.Params(M.MODEL_BGK, 0.8, 0.0, 1e-5, 0.0)) for _ in range(2))
    assert (RECORDS in _kernels(lambda: M.step(ctx, 2))) == large
    M.set_kernel_variant(ref, 0)
    assert RECORDS not in _kernels(lambda: M.step(ref, 2))
    assert np.array_equal(M.get_populations(ctx), M.get_populations(ref))
