"""The step kernels whose warps stream 32-node tiles through shared-memory
slots of their own (variants 27-29): tile edges, link nodes next to plain ones
in a warp, kinds that change under a batch's run to steady state, and the tile
ranges on sets of mixed kinds.  The elementwise comparison with the oracle is
in test_gpu_parity (every variant)."""
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


def _state(M, ctx):
    return M.get_populations(ctx) if ctx.model == M.MODEL_BGK else M.get_fields(ctx)


# node counts around one tile, several tiles, and one tile per block of the grid
@pytest.mark.parametrize("nx,ny", [(8, 4), (11, 3), (21, 3), (13, 5), (32, 33), (139, 35)])
@pytest.mark.parametrize("K", [12, 16, 24, 32])
@pytest.mark.parametrize("model", ["bgk", "tau1"])
def test_tile_edges_match_the_plain_kernel(M, nx, ny, K, model):
    w = I.poiseuille_channel(nx, ny, 0.2, seed=4)
    if w.n < K:
        pytest.skip("fewer nodes than the stencil")
    st = M.build_stencils_for(w, K=K, s=0.5, bb_mode=M.BB_INTERPOLATED)
    p = M.Params(M.MODEL_BGK, 0.8, 1.1, 1e-5, 0.0) if model == "bgk" else M.Params(M.MODEL_TAU1, 1.0, 0.0, 1e-5, 0.0)
    out = {}
    for v in (0, 27, 28, 29):
        ctx = M.init(st, p)
        M.set_kernel_variant(ctx, v)
        M.set_fields(ctx, _start(w))
        M.step(ctx, 5)
        out[v] = _state(M, ctx)
    # five steps; a step's interpolated values are sums of at most 31 products
    # of weights of magnitude <= ~2 and differences <= ~0.05, formed in another
    # order: (31 + 20) 2^-24 * 0.1 per step is 3e-7
    for v in (27, 28, 29):
        assert np.isfinite(out[v]).all()
        assert np.abs(out[v] - out[0]).max() < 5 * 3e-7


@pytest.mark.parametrize("bounds", [None, "uneven"])
def test_a_nodes_result_does_not_depend_on_its_warp(M, bounds):
    """Ranges that cut the tiles elsewhere put link nodes and plain nodes into
    other warps: bitwise the same step."""
    w = I.porous(seed=6, n_target=4000)
    st = M.build_stencils_for(w, K=16, s=0.5, bb_mode=M.BB_INTERPOLATED)
    b = None if bounds is None else [0, 37, 1501, w.n]
    for p in (M.Params(M.MODEL_BGK, 0.8, 1.1, 1e-6, 0.0), M.Params(M.MODEL_TAU1, 1.0, 0.0, 1e-6, 0.0)):
        ref, part = M.init(st, p), M.Partitioned(st, p, 3, b)
        for v in (27, 28):
            M.set_kernel_variant(ref, v)
            part.set_kernel_variant(v)
            M.set_fields(ref, _start(w))
            part.set_fields(_start(w))
            M.step(ref, 7)
            part.step(7)
            assert np.array_equal(part.get_fields(), M.get_fields(ref))


def test_held_samples_of_a_batch(M):
    """Samples held at their steady state change their kinds in the tile
    records while the run goes on, across tiles that two samples share, and
    the kinds come back: the batch then steps like a fresh one."""
    ws = [I.porous(seed=s, n_target=n) for s, n in ((1, 1500), (2, 2300), (3, 900))]
    sts = [M.build_stencils_for(w, K=16, s=1.0) for w in ws]
    ps = [M.Params(M.MODEL_TAU1, 1.0, 0.0, g, 0.0) for g in (1e-6, 5e-6, 2e-6)]
    batch = M.batch_init(sts, ps)
    assert M.kernel_variant(batch) == 27
    steps = M.batch_run_to_steady(batch, 1e-6, 200, 20000, check=50)
    fields = M.get_fields(batch)
    assert len(set(steps.tolist())) > 1
    for i, (st, p) in enumerate(zip(sts, ps)):
        one = M.init(st, p)
        assert M.run_to_steady(one, 1e-6, 200, 20000, check=50) == steps[i]
        a, n = M.batch_range(batch, i)
        assert np.array_equal(M.get_fields(one), fields[a:a + n])
    fresh = M.batch_init(sts, ps)
    start = np.concatenate([_start(w) for w in ws])
    for c in (batch, fresh):
        M.set_fields(c, start)
        M.step(c, 33)
    assert np.array_equal(M.get_fields(batch), M.get_fields(fresh))


def test_mixed_kinds_over_the_ranges(M):
    """Equilibrium, Lagrange and scattered tiles in one set, more tiles than
    blocks: every node is stepped once, as by the plain kernel."""
    w = I.karman(scale=0.3, lattice_beyond_d=1.0, areas="spacing")
    st = M.build_stencils_for(w, K=16, s=0.5, bb_mode=M.BB_SIMPLE)
    out = {}
    for v in (0, 27):
        ctx = M.init(st, M.Params(M.MODEL_BGK, 0.7, 0.0, 0.0, 0.0))
        M.set_kernel_variant(ctx, v)
        M.set_fields(ctx, _start(w))
        M.step(ctx, 6)
        out[v] = M.get_populations(ctx)
    assert np.abs(out[27] - out[0]).max() < 6 * 3e-7


@pytest.mark.parametrize("n_parts", [1, 7, 40])
@pytest.mark.parametrize("model", ["bgk", "tau1"])
def test_partitions_in_one_launch(M, n_parts, model):
    """All ranges in one launch that stores the halo states itself: bitwise the
    unpartitioned step over graph replays and single steps, for more ranges
    than a small set has tiles per range, and after changing the variant."""
    w = I.porous(seed=8, n_target=3000)
    st = M.build_stencils_for(w, K=16, s=1.0)
    p = M.Params(M.MODEL_BGK, 0.8, 0.0, 1e-6, 0.0) if model == "bgk" else M.Params(M.MODEL_TAU1, 1.0, 0.0, 1e-6, 0.0)
    ref, part = M.init(st, p), M.Partitioned(st, p, n_parts)
    for n, v in ((1, 27), (35, 27), (17, 11), (16, 29)):
        M.set_kernel_variant(ref, v)
        part.set_kernel_variant(v)
        if v == 27:
            M.set_fields(ref, _start(w))
            part.set_fields(_start(w))
        M.step(ref, n)
        part.step(n)
        assert np.array_equal(part.get_fields(), M.get_fields(ref)), (n, v)
