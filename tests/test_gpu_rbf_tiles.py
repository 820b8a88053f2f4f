"""The BGK step from tile records of RBF-FD weights against the plain RBF-FD
kernel, which reads every weight: the records leave out zeros and keep the slot
order, so the states agree bit for bit -- at the edges of a tile, with links of
both rules, Lagrange and equilibrium nodes in a tile, stencils per Lagrangian
point of several sizes, batches and partitions.  Variant 28 takes the records at
any size; large sets of stencils per Lagrangian point take them by default."""
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


def _start(w):
    x, y = w.xy[:, 0], w.xy[:, 1]
    return np.stack([1 + 1e-3 * np.sin(x / 7), 0.02 * np.sin(y / 5 + 1), 0.01 * np.cos(x / 6)], 1)


def _pair(M, st, w, steps, variant=28):
    out = []
    for v in (0, variant):
        ctx = M.init(st, M.Params(M.MODEL_BGK, 0.8, 1.1, 1e-5, 0.0))
        M.set_kernel_variant(ctx, v)
        M.set_fields(ctx, _start(w))
        M.step(ctx, steps)
        out.append(M.get_populations(ctx))
    assert np.isfinite(out[0]).all()
    return out


@pytest.mark.parametrize("nx,ny", [(8, 5), (11, 3), (16, 3), (21, 13), (139, 35)])
@pytest.mark.parametrize("K,n_l,bb", [(12, 0, 1), (24, 0, 1), (32, 0, 0), (32, 7, 0), (32, 7, 1)])
def test_tile_edges(M, nx, ny, K, n_l, bb):
    w = I.poiseuille_channel(nx, ny, 0.2, seed=4)
    if w.n < max(K, n_l):
        pytest.skip("fewer nodes than the stencil")
    kw = {"interp": M.INTERP_RBF_POINTS, "n_l": n_l} if n_l else {"interp": M.INTERP_RBF}
    st = M.build_stencils_for(w, K=K, s=0.5, bb_mode=bb, **kw)
    a, b = _pair(M, st, w, 19)  # a replayed graph and single steps
    assert np.array_equal(a, b)


@pytest.mark.parametrize("hybrid", [False, True])
def test_mixed_kinds(M, hybrid):
    w = I.karman(scale=0.2, seed=3, lattice_beyond_d=1.0 if hybrid else None, areas="spacing")
    st = M.build_stencils_for(w, K=24, s=0.5, bb_mode=M.BB_INTERPOLATED, interp=M.INTERP_RBF)
    a, b = _pair(M, st, w, 6)
    assert np.array_equal(a, b)


@pytest.mark.parametrize("bb", [0, 1])
def test_default_of_a_large_set(M, bb):
    w = I.poiseuille_channel(300, 157, 0.2, seed=4)  # 47,100 nodes of 2.3 KB
    st = M.build_stencils_for(w, K=64, s=0.5, bb_mode=bb, interp=M.INTERP_RBF_POINTS, n_l=25)
    a, b = _pair(M, st, w, 19, variant=1)
    assert np.array_equal(a, b)


def test_batch_and_partitions(M):
    ws = [I.porous(seed=s, n_target=n) for s, n in ((1, 1500), (2, 2301))]
    sts = [M.build_stencils_for(w, K=24, s=0.5, interp=M.INTERP_RBF) for w in ws]
    ps = [M.Params(M.MODEL_BGK, 0.8, 0.0, 1e-6, 0.0), M.Params(M.MODEL_BGK, 0.9, 1.0, 2e-6, 0.0)]
    batch = M.batch_init(sts, ps)
    M.set_kernel_variant(batch, 28)
    M.set_fields(batch, np.concatenate([_start(w) for w in ws]))
    M.step(batch, 20)
    got = M.get_fields(batch)
    for i, (w, st, p) in enumerate(zip(ws, sts, ps)):
        ref, part = M.init(st, p), M.Partitioned(st, p, 3)
        M.set_kernel_variant(ref, 0)
        part.set_kernel_variant(28)
        M.set_fields(ref, _start(w))
        part.set_fields(_start(w))
        M.step(ref, 20)
        part.step(20)
        want = M.get_fields(ref)
        a, n = M.batch_range(batch, i)
        assert np.array_equal(got[a:a + n], want)
        assert np.array_equal(part.get_fields(), want)
