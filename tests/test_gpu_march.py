"""Two steps per launch (the march, csrc/lbm_march.cuh) against one step per
launch: the march forms every value by the one-step kernels' functions, so an
AUTO lattice, which marches on grids of these sizes, has a GENERIC lattice's
bits.  Sizes at the edges of the strips (up to 122 columns) and of the chunks of
rows, one strip only, narrow and odd grids, every storage format and boundary,
both normals, odd step counts and checks that fall between steps; a few of them
through the index-checking build as well."""
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


def _run(lbm, nx, ny, bc, storage, steps, kernel, normal=0, check_every=0):
    P = dict(rho_l=1.0, rho_g=0.01, nu_l=0.05, nu_g=0.1, visc_mode=0, sigma=1e-3, W=4.0, tau_h=0.8,
             Gx=1e-6, Gy=-2e-6, bc_y=bc, normal_scheme=normal, check_every=check_every)
    phi0 = cases.spinodal(nx, ny, 0.5, 0.2, seed=nx + ny)
    ux0 = 1e-3 * (cases.spinodal(nx, ny, 0.0, 1.0, seed=7))
    with lbm.Lattice(nx, ny, storage=storage, kernel=kernel, **P) as g:
        g.init(phi0, ux0)
        for n in steps:
            g.step(n)
        return (*g.get_state(), *g.fields().values())


def _same(a, b):
    assert np.isfinite(a[0]).all()
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


SIZES = [(701, 333), (732, 456), (733, 457), (122, 2500), (123, 4700), (64, 13000), (1001, 778), (2400, 300)]


@pytest.mark.parametrize("storage", [0, 1, 2, 3])
@pytest.mark.parametrize("bc", [0, 1, 2])
def test_march_equals_single_steps(libs, storage, bc):
    lbm, release, _ = libs
    lbm._LIB_PATH, lbm._lib = release, None
    for nx, ny in SIZES:
        _same(_run(lbm, nx, ny, bc, storage, (7, 2, 4), 0), _run(lbm, nx, ny, bc, storage, (7, 2, 4), 1))


@pytest.mark.parametrize("normal,check_every", [(1, 0), (0, 1), (0, 3), (1, 4)])
def test_march_options(libs, normal, check_every):
    lbm, release, _ = libs
    lbm._LIB_PATH, lbm._lib = release, None
    for storage, bc in ((0, 0), (1, 2), (0, 1)):
        _same(_run(lbm, 801, 600, bc, storage, (11,), 0, normal, check_every),
              _run(lbm, 801, 600, bc, storage, (11,), 1, normal, check_every))


def test_march_reports_a_nonfinite_node(libs):
    lbm, release, _ = libs
    lbm._LIB_PATH, lbm._lib = release, None
    nx, ny = 900, 700
    for bad in ((0, 0), (ny - 1, nx - 1), (350, 123)):
        with lbm.Lattice(nx, ny, check_every=4, **cases.params_spinodal()) as g:
            g.init(cases.spinodal(nx, ny)).step(4)
            f, gg, pu = (a.copy() for a in g.get_state())
            gg[3][bad] = np.nan
            g.set_state(f, gg, pu)
            g.step(2)
            with pytest.raises(lbm.LbmError) as e:
                g.step(2)
            assert e.value.status == lbm.LBM_ERR_NONFINITE


@pytest.mark.parametrize("storage", [0, 2])
def test_march_in_the_checking_build(libs, storage):
    lbm, release, debug = libs
    for nx, ny, bc in ((733, 457, 0), (732, 456, 2), (701, 333, 1)):
        got = []
        for path in (debug, release):
            lbm._LIB_PATH, lbm._lib = path, None
            got.append(_run(lbm, nx, ny, bc, storage, (9,), 0, 0, 3))
        _same(*got)


def _batch(lbm, n, storage, kernel, steps, check_every=0):
    specs = cases.batch_cases(n, seed=11)
    specs[3]["params"] = dict(specs[3]["params"], bc_y=2)
    lats = [lbm.Lattice(sp["nx"], sp["ny"], storage=storage, kernel=kernel, check_every=check_every, **sp["params"])
            .init(sp["phi0"], sp["ux0"], sp["uy0"]) for sp in specs]
    try:
        with lbm.Batch(lats) as bt:
            for k in steps:
                bt.step(k)
                lats[2].step(3)  # a case stepped on its own in between
        return [a for lat in lats for a in lat.get_state()]
    finally:
        for lat in lats:
            lat.close()


@pytest.mark.parametrize("n,storage,check_every", [(16, 0, 0), (16, 0, 1), (36, 1, 0), (36, 2, 2)])
def test_batch_march_equals_single_steps(libs, n, storage, check_every):
    """Batches large enough to march: fewer steps than a graph, odd counts, the
    tuning call, graph replays with even and odd remainders."""
    lbm, release, debug = libs
    steps = (7, 4, 1, 151, 67, 34)
    lbm._LIB_PATH, lbm._lib = release, None
    got = _batch(lbm, n, storage, 0, steps, check_every)
    _same(got, _batch(lbm, n, storage, 1, steps, check_every))
    if check_every:
        lbm._LIB_PATH, lbm._lib = debug, None
        _same(_batch(lbm, n, storage, 0, steps, check_every), got)
