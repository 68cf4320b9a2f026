"""Several steps per launch of small grids (csrc/lbm_tile.cuh) against one step
per launch: every value is formed by the one-step kernels' functions, so an AUTO
lattice of these sizes has a GENERIC lattice's bits.  One-node and one-tile
grids (whose halo wraps several times), narrow and ragged ones, every storage
format and boundary, both normals, step counts that leave every remainder, and
checks that fall between steps; also through the index-checking build."""
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
    P = dict(rho_l=1.0, rho_g=0.1, nu_l=0.1, nu_g=0.1, visc_mode=2, sigma=1e-3, W=3.0, tau_h=0.8, Gx=1e-5, Gy=2e-5,
             bc_y=bc, normal_scheme=normal, check_every=check_every)
    r = np.random.default_rng(100 * nx + ny)
    phi0, ux0 = 0.5 + 0.3 * r.random((ny, nx)), 1e-3 * r.standard_normal((ny, nx))
    with lbm.Lattice(nx, ny, storage=storage, kernel=kernel, **P) as g:
        g.init(phi0, ux0)
        for n in steps:
            g.step(n)
        return (*g.get_state(), *g.fields().values())


def _same(a, b):
    assert np.isfinite(a[0]).all()
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


SIZES = [(2, 2), (3, 5), (5, 2), (2, 200), (200, 3), (8, 256), (9, 9), (31, 17), (64, 64), (65, 63), (128, 128),
         (133, 97), (200, 200), (211, 190)]


@pytest.mark.parametrize("storage", [0, 1, 2, 3])
@pytest.mark.parametrize("bc", [0, 1, 2])
def test_tiles_equal_single_steps(libs, storage, bc):
    lbm, release, _ = libs
    lbm._LIB_PATH, lbm._lib = release, None
    for nx, ny in SIZES:
        steps = (13, 1, 2, 3, 4, 6, 10)
        _same(_run(lbm, nx, ny, bc, storage, steps, 0), _run(lbm, nx, ny, bc, storage, steps, 1))


@pytest.mark.parametrize("normal,check_every", [(1, 0), (0, 1), (0, 3), (1, 5)])
def test_tile_options(libs, normal, check_every):
    lbm, release, _ = libs
    lbm._LIB_PATH, lbm._lib = release, None
    for storage, bc in ((0, 0), (1, 2), (0, 1)):
        _same(_run(lbm, 70, 45, bc, storage, (23,), 0, normal, check_every),
              _run(lbm, 70, 45, bc, storage, (23,), 1, normal, check_every))


def test_tiles_report_a_nonfinite_node(libs):
    lbm, release, _ = libs
    lbm._LIB_PATH, lbm._lib = release, None
    for bad in ((0, 0), (63, 63), (30, 17)):
        with lbm.Lattice(64, 64, check_every=8, **cases.params_static_drop()) as g:
            g.init(cases.drop(64, 64, 16, 4.0)).step(8)
            f, gg, pu = (a.copy() for a in g.get_state())
            gg[3][bad] = np.nan
            g.set_state(f, gg, pu)
            g.step(4)
            with pytest.raises(lbm.LbmError) as e:
                g.step(4)
            assert e.value.status == lbm.LBM_ERR_NONFINITE


@pytest.mark.parametrize("storage", [0, 2])
def test_tiles_in_the_checking_build(libs, storage):
    lbm, release, debug = libs
    for nx, ny, bc in ((64, 64, 0), (3, 5, 0), (33, 20, 2), (8, 100, 1)):
        got = []
        for path in (debug, release):
            lbm._LIB_PATH, lbm._lib = path, None
            got.append(_run(lbm, nx, ny, bc, storage, (17,), 0, 0, 3))
        _same(*got)
