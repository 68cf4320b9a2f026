"""Steps under stream capture: a graph of an even number of lbm_step or
lbm_batch_step steps, replayed, advances the state as direct one-step launches
(LBM_KERNEL_GENERIC) do, bit for bit, on grids where the library otherwise takes
several steps per launch; also with plain steps, a restore or an initialisation
between the replays."""
import numpy as np
import pytest

from paper_1710_09541_gb300 import cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09541_gb300 import build as lbm_build
    from paper_1710_09541_gb300 import lbm as _lbm

    lbm_build.build()
    _lbm.load()
    return _lbm, torch


def _lattice(lbm, nx, ny, storage, bc, kernel, stream):
    P = dict(cases.params_spinodal(), bc_y=bc)
    return lbm.Lattice(nx, ny, stream=stream, storage=storage, kernel=kernel, **P).init(cases.spinodal(nx, ny))


def _same(a, b):
    assert np.isfinite(a[0]).all()
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def _capture(torch, stream, fn):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=stream):
        fn()
    torch.cuda.synchronize()
    return g


def _replay(torch, stream, g, n):
    with torch.cuda.stream(stream):
        for _ in range(n):
            g.replay()
    torch.cuda.synchronize()


# 64 x 64 and 33 x 50: tiles; 801 x 600 and 1280 x 1280: the march (every format)
@pytest.mark.parametrize("nx,ny,storage,bc", [(64, 64, 0, 0), (33, 50, 2, 1), (801, 600, 0, 0), (801, 600, 1, 2),
                                              (1280, 1280, 0, 0)])
@pytest.mark.parametrize("before", [0, 2, 3])
@pytest.mark.parametrize("n", [2, 6])
def test_captured_steps_replay(env, nx, ny, storage, bc, before, n):
    lbm, torch = env
    s = torch.cuda.Stream()
    with _lattice(lbm, nx, ny, storage, bc, 0, s) as a, _lattice(lbm, nx, ny, storage, bc, 1, s) as b:
        a.step(before)
        b.step(before)
        g = _capture(torch, s, lambda: a.step(n))
        _replay(torch, s, g, 3)
        b.step(3 * n)
        _same(a.get_state(), b.get_state())
        a.step(4)                       # plain steps between replays
        _replay(torch, s, g, 1)
        b.step(4 + n)
        _same((*a.get_state(), *a.fields().values()), (*b.get_state(), *b.fields().values()))
        if before % 2 == 0:             # init and restore start from buffer 0
            state = [x.copy() for x in b.get_state()]
            a.init(cases.spinodal(nx, ny))
            _replay(torch, s, g, 2)
            b.init(cases.spinodal(nx, ny)).step(2 * n)
            _same(a.get_state(), b.get_state())
            a.set_state(*state)
            _replay(torch, s, g, 2)
            b.set_state(*state).step(2 * n)
            _same(a.get_state(), b.get_state())
        del g


@pytest.mark.parametrize("before", [0, 2, 34])
def test_captured_batch_steps_replay(env, before):
    """16 cases, enough for the batch's two-step launches."""
    lbm, torch = env
    s = torch.cuda.Stream()
    specs = cases.batch_cases(16, seed=11)

    def make(kernel):
        return [lbm.Lattice(sp["nx"], sp["ny"], stream=s, kernel=kernel, **sp["params"])
                .init(sp["phi0"], sp["ux0"], sp["uy0"]) for sp in specs]

    A, B = make(0), make(1)
    try:
        with lbm.Batch(A) as bt, lbm.Batch(B) as ref:
            bt.step(before)
            for lat in A[:8]:           # moves some cases' buffers
                lat.step(2)
            g = _capture(torch, s, lambda: bt.step(6))
            _replay(torch, s, g, 3)
            bt.step(34)
            A[2].step(4)
            _replay(torch, s, g, 1)
            ref.step(before + 18 + 34)
            for lat in B[:8]:
                lat.step(2)
            B[2].step(4)
            ref.step(6)
            for a, b in zip(A, B):
                _same(a.get_state(), b.get_state())
            del g
    finally:
        for lat in A + B:
            lat.close()
