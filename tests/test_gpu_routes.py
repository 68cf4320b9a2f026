"""Which kernels the library's rules choose, by the launches they count, and the
routes that no other test's sizes take.  A comparison of LBM_KERNEL_AUTO with
LBM_KERNEL_GENERIC says something only where the two take different kernels, so
each one here first asserts how many steps AUTO took per launch."""
import numpy as np
import pytest

from paper_1710_09541_gb300 import cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def libs():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1710_09541_gb300 import build as lbm_build
    from paper_1710_09541_gb300 import lbm

    release, debug = lbm_build.build(), lbm_build.build(debug=True)
    saved = (lbm._LIB_PATH, lbm._lib)
    yield lbm, release, debug
    lbm._LIB_PATH, lbm._lib = saved


def _use(lbm, path):
    lbm._LIB_PATH, lbm._lib = path, None


def _same(a, b):
    assert np.isfinite(a[0]).all()
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def _run(lbm, nx, ny, bc, storage, steps, kernel):
    P = dict(rho_l=1.0, rho_g=0.01, nu_l=0.05, nu_g=0.1, visc_mode=0, sigma=1e-3, W=4.0, tau_h=0.8,
             Gx=1e-6, Gy=-2e-6, bc_y=bc)
    with lbm.Lattice(nx, ny, storage=storage, kernel=kernel, **P) as g:
        g.init(cases.spinodal(nx, ny, 0.5, 0.2, seed=nx + ny), 1e-3 * cases.spinodal(nx, ny, 0.0, 1.0, seed=7))
        g.step(steps)
        return g.step_launches(), [*g.get_state(), *g.fields().values()]


# one narrow strip; a low and wide grid; rows of whole sectors in every format
MARCHING = [(65, 9000, 0), (67, 20000, 1), (67, 20000, 2), (67, 20000, 3), (20001, 16, 0), (20001, 16, 1),
            (1280, 1280, 0), (1280, 1280, 1), (1280, 1280, 2), (1280, 1280, 3), (701, 333, 0), (123, 4700, 0)]


@pytest.mark.parametrize("nx,ny,storage", MARCHING)
@pytest.mark.parametrize("bc", [0, 1, 2])
def test_march_where_it_is_chosen(libs, nx, ny, storage, bc):
    lbm, release, _ = libs
    _use(lbm, release)
    n, got = _run(lbm, nx, ny, bc, storage, 9, 0)
    assert n == 5  # four pairs and one step
    m, want = _run(lbm, nx, ny, bc, storage, 9, 1)
    assert m == 9
    _same(got, want)


@pytest.mark.parametrize("nx,ny,storage,per_launch", [(64, 64, 0, 3), (8, 256, 0, 3), (200, 200, 2, 2), (3, 5, 1, 4),
                                                      (1, 64, 0, 1), (512, 512, 0, 1), (1024, 1024, 1, 1)])
def test_steps_per_launch(libs, nx, ny, storage, per_launch):
    lbm, release, _ = libs
    _use(lbm, release)
    n, got = _run(lbm, nx, ny, 0, storage, 12, 0)
    assert n == 12 // per_launch
    if per_launch > 1:
        _same(got, _run(lbm, nx, ny, 0, storage, 12, 1)[1])


# 8.7 M nodes in strips close to 122 columns, so that 16-bit batches march; both classes
LARGE = [(976, 960, 0), (976, 960, 1), (1098, 801, 0), (1220, 640, 2), (973, 1100, 0), (976, 720, 1), (610, 1300, 0),
         (1097, 900, 1), (976, 960, 2), (366, 1500, 0)]


def _batch(lbm, specs, storage, kernel, steps, check_every=0):
    lats = []
    for nx, ny, bc in specs:
        P = dict(cases.params_spinodal(), bc_y=bc, check_every=check_every)
        lats.append(lbm.Lattice(nx, ny, storage=storage, kernel=kernel, **P).init(cases.spinodal(nx, ny, seed=nx + ny)))
    try:
        with lbm.Batch(lats) as bt:
            counts = []
            for k in steps:
                bt.step(k)
                counts.append(bt.counts()[0])
                lats[2].step(3)  # a case stepped on its own in between
        return counts, [a for lat in lats for a in lat.get_state()]
    finally:
        for lat in lats:
            lat.close()


@pytest.mark.parametrize("storage,check_every", [(1, 0), (2, 0), (1, 2), (2, 1)])
def test_16bit_batch_march(libs, storage, check_every):
    """Fewer steps than a graph, odd counts, graph replays with even and odd
    remainders; with checks also through the index-checking build."""
    lbm, release, debug = libs
    steps = (7, 4, 1, 67, 34)
    _use(lbm, release)
    n, got = _batch(lbm, LARGE, storage, 0, steps, check_every)
    assert n == [8, 12, 14, 82, 116]  # per class: 3 + 1, 2, 1, 32 + 1 + 1, 16 + 1
    m, want = _batch(lbm, LARGE, storage, 1, steps, check_every)
    assert m[-1] == 2 * sum(steps)
    _same(got, want)
    if check_every:
        _use(lbm, debug)
        n, again = _batch(lbm, LARGE, storage, 0, steps, check_every)
        assert n[-1] == 116
        _same(again, want)


@pytest.mark.parametrize("odd", [False, True])
def test_prefetching_batch_steps(libs, odd):
    """One-step launches of a 16-bit batch above the prefetch threshold (tensor
    maps; with one more case of nx = 1004 per-thread requests) against cases
    stepped alone: the two-step launches leave this path only to GENERIC cases
    and to batches below their own threshold."""
    lbm, release, _ = libs
    _use(lbm, release)
    specs = cases.batch_cases(24, seed=11)  # 6 M nodes: 552 MB a step
    if odd:
        phi0 = cases.drop(1004, 300, 40.0, 4.0)
        specs.append(dict(nx=1004, ny=300, params=cases.params_static_drop(ratio=100.0), phi0=phi0, ux0=None, uy0=None))
    pick = [0, 1, 23, len(specs) - 1]

    def make(which, kernel):
        return [lbm.Lattice(sp["nx"], sp["ny"], storage=1, kernel=kernel, **sp["params"])
                .init(sp["phi0"], sp["ux0"], sp["uy0"]) for sp in which]

    A, B = make(specs, 1), make([specs[k] for k in pick], 1)
    try:
        with lbm.Batch(A) as bt:
            bt.step(10)
            assert bt.counts()[0] == 20
        for lat in B:
            lat.step(10)
        for k, b in zip(pick, B):
            _same(A[k].get_state(), b.get_state())
    finally:
        for lat in A + B:
            lat.close()


@pytest.mark.parametrize("storage,pairs", [(0, True), (1, False)])
def test_first_long_batch_call(libs, storage, pairs):
    """The first call of 140 or more steps times what the batch runs: pairs of
    steps (no one-step launch then), or the tile shapes."""
    lbm, release, _ = libs
    _use(lbm, release)
    specs = cases.batch_cases(16, seed=11)
    lats = [lbm.Lattice(sp["nx"], sp["ny"], storage=storage, **sp["params"]).init(sp["phi0"], sp["ux0"], sp["uy0"])
            for sp in specs]
    alone = [lbm.Lattice(sp["nx"], sp["ny"], storage=storage, kernel=lbm.LBM_KERNEL_GENERIC, **sp["params"])
             .init(sp["phi0"], sp["ux0"], sp["uy0"]).step(161) for sp in specs[:3]]
    try:
        with lbm.Batch(lats) as bt:
            assert not bt.info()["tuned"]
            bt.step(161)
            assert bt.counts()[0] == 2 * (81 if pairs else 161)
            info = bt.info()
            assert info["tuned"] and info["periodic"]["us"] > 0 and info["walls"]["us"] > 0
        for a, b in zip(lats, alone):
            _same(a.get_state(), b.get_state())
    finally:
        for lat in lats + alone:
            lat.close()


@pytest.mark.parametrize("storage,n", [(0, 50), (0, 47), (1, 33)])
def test_batch_graphs_are_kept(libs, storage, n):
    """Calls that leave the state in other buffers than they found it in (50: an
    odd number of pairs, 47: of pairs and a step, 33: of single steps) replay one
    graph per starting buffer; a case stepped on its own makes new ones."""
    lbm, release, _ = libs
    _use(lbm, release)
    specs = cases.batch_cases(8, seed=11)

    def make(kernel):
        return [lbm.Lattice(sp["nx"], sp["ny"], storage=storage, kernel=kernel, **sp["params"])
                .init(sp["phi0"], sp["ux0"], sp["uy0"]) for sp in specs]

    A, B = make(0), make(1)
    try:
        with lbm.Batch(A) as bt:
            for _ in range(8):
                bt.step(n)
            assert bt.counts()[1] == {50: 2, 47: 2, 33: 2}[n]
            for lat in B:
                lat.step(8 * n)
            for a, b in zip(A, B):
                _same(a.get_state(), b.get_state())
            A[3].step(1)
            B[3].step(1)
            for _ in range(5):
                bt.step(n)
            assert bt.counts()[1] == 4
            for lat in B:
                lat.step(5 * n)
            for a, b in zip(A, B):
                _same((*a.get_state(), *a.fields().values()), (*b.get_state(), *b.fields().values()))
    finally:
        for lat in A + B:
            lat.close()


def test_batch_prefetch_follows_the_phiu_buffer(libs):
    """The index-checking build also checks that each prefetch map of a one-step
    16-bit batch covers the buffer about to be read.  A several-step launch of one
    case alone moves its (phi u) to the other buffer."""
    lbm, release, debug = libs
    _use(lbm, debug)
    specs = cases.batch_cases(24, seed=11)
    P = cases.params_static_drop()
    specs.append(dict(nx=64, ny=64, params=P, phi0=cases.drop(64, 64, 16.0, P["W"]), ux0=None, uy0=None))
    A = [lbm.Lattice(sp["nx"], sp["ny"], storage=1, check_every=1 << 20, **sp["params"])
         .init(sp["phi0"], sp["ux0"], sp["uy0"]) for sp in specs]
    try:
        with lbm.Batch(A) as bt:
            bt.step(3)
            assert bt.counts()[0] == 6
            A[24].step(3)
            assert A[24].step_launches() == 1
            bt.step(4)
            A[24].init(specs[24]["phi0"])
            bt.step(33)
    finally:
        for lat in A:
            lat.close()


def test_bench_bytes_per_update_follow_the_launches(libs):
    """bench.py's bytes per update of a batch are those of the launches it made:
    half of a step's where the batch takes pairs (FP32 here), a whole step's
    where it takes one-step launches."""
    import torch

    import bench

    lbm, release, _ = libs
    _use(lbm, release)
    full = cases.batch_cases
    cases.batch_cases = lambda n=64, seed=11: full(8, seed=11)
    try:
        s = torch.cuda.current_stream()
        for storage, launches, bytes_ in ((0, 1.0, 80.0), (1, 2.0, 92.0)):
            d = bench.run_batched(torch, lbm, s, 40, storage=storage)
            assert d["cases"] == 8 and d["launches_per_step"] == launches and d["bytes_per_lu"] == bytes_
    finally:
        cases.batch_cases = full
