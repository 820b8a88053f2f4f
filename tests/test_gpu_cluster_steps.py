"""Runs by one cluster that keeps the set in shared memory (variant 27, small
sets) against one launch per step: bitwise the same state, for sets of less
than a tile, fewer tiles than blocks, the last block without tiles, the largest
that fit and the first that do not, odd and even step counts, all kinds of
nodes, batches, and several contexts at once."""
import threading

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


def _params(M):
    return M.Params(M.MODEL_BGK, 0.8, 1.1, 1e-5, 0.0)


def _both(M, st, p, start, counts):
    out = []
    for graphs in (False, True):  # without graphs every step is a launch
        ctx = M.init(st, p)
        M.set_graphs(ctx, graphs)
        M.set_fields(ctx, start)
        for n in counts:
            M.step(ctx, n)
        out.append(M.get_populations(ctx))
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("nx,ny", [(8, 4), (11, 3), (21, 13), (32, 33), (97, 20), (64, 31), (64, 32), (49, 42)])
@pytest.mark.parametrize("K", [12, 16, 24, 32])
def test_matches_a_launch_per_step(M, nx, ny, K):
    w = I.poiseuille_channel(nx, ny, 0.2, seed=4)
    if w.n < K:
        pytest.skip("fewer nodes than the stencil")
    st = M.build_stencils_for(w, K=K, s=0.5, bb_mode=M.BB_INTERPOLATED)
    _both(M, st, _params(M), _start(w), (8, 3, 17))


@pytest.mark.parametrize("bb", [0, 1])
def test_mixed_kinds(M, bb):
    w = I.karman(scale=0.1, lattice_beyond_d=1.0, areas="spacing")
    st = M.build_stencils_for(w, K=16, s=0.5, bb_mode=bb)
    _both(M, st, _params(M), _start(w), (9,))


def test_batch(M):
    ws = [I.porous(seed=s, n_target=n) for s, n in ((1, 700), (2, 1100))]
    sts = [M.build_stencils_for(w, K=16, s=1.0) for w in ws]
    ps = [M.Params(M.MODEL_BGK, 0.7, 0.0, 1e-6, 0.0), M.Params(M.MODEL_BGK, 0.9, 1.2, 0.0, 5e-6)]
    got = []
    for graphs in (False, True):
        b = M.batch_init(sts, ps)
        M.set_graphs(b, graphs)
        M.set_fields(b, np.concatenate([_start(w) for w in ws]))
        M.step(b, 33)
        got.append(M.get_populations(b))
    assert np.array_equal(*got)


def test_contexts_at_once(M):
    """Runs on streams of their own from two threads."""
    w = I.porous(seed=6, n_target=1900)
    st = M.build_stencils_for(w, K=16, s=1.0)
    p = _params(M)
    ref = M.init(st, p)
    M.set_fields(ref, _start(w))
    M.set_graphs(ref, False)
    M.step(ref, 1200)
    want = M.get_fields(ref)
    out = [None, None]

    def go(i):
        ctx = M.init(st, p)
        M.set_fields(ctx, _start(w))
        for _ in range(60):
            M.step(ctx, 20)
        out[i] = M.get_fields(ctx)

    threads = [threading.Thread(target=go, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert all(np.array_equal(o, want) for o in out)
