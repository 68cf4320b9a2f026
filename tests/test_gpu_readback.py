"""lbm_get_fields into page-locked host memory, which the read-back kernel writes
itself, against pageable memory, which the copies fill: the same bits for whole
allocations, parts of one, registered memory, some outputs only, mixed kinds and
overlapping outputs; nothing outside the outputs is written."""
import ctypes

import numpy as np
import pytest

from paper_1710_09541_gb300 import cases

pytestmark = pytest.mark.gpu
KEYS = ("phi", "rho", "ux", "uy", "p")


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


@pytest.mark.parametrize("nx,ny,bc,storage", [(1, 2, 0, 0), (33, 17, 1, 1), (500, 301, 2, 0), (64, 64, 0, 3)])
def test_pinned_outputs(env, nx, ny, bc, storage):
    lbm, torch = env
    P = dict(cases.params_static_drop(ratio=100.0), bc_y=bc)
    n = nx * ny
    with lbm.Lattice(nx, ny, storage=storage, **P) as a:
        a.init(cases.drop(nx, ny, 0.3 * min(nx, ny) + 1, 4.0)).step(5)
        want = a.fields()
        buf = torch.full((5 * n + 7,), -7.0, dtype=torch.float64, pin_memory=True)
        flat = buf.numpy()
        out = {k: flat[3 + j * n:3 + (j + 1) * n].reshape(ny, nx) for j, k in enumerate(KEYS)}
        a.fields(out=out)
        for k in KEYS:
            assert np.array_equal(out[k], want[k]), k
        assert (flat[:3] == -7.0).all() and (flat[3 + 5 * n:] == -7.0).all()
        # some outputs only, straight through the C ABI
        flat[:] = -7.0
        ptr = ctypes.POINTER(ctypes.c_double)
        a._check(a._L.lbm_get_fields(a._h, None, None, out["ux"].ctypes.data_as(ptr), None,
                                     out["p"].ctypes.data_as(ptr)))
        assert np.array_equal(out["ux"], want["ux"]) and np.array_equal(out["p"], want["p"])
        assert (out["phi"] == -7.0).all() and (out["uy"] == -7.0).all()
        # pinned and pageable together
        mixed = {k: (out[k] if j % 2 else np.empty((ny, nx))) for j, k in enumerate(KEYS)}
        a.fields(out=mixed)
        for k in KEYS:
            assert np.array_equal(mixed[k], want[k]), k
        # overlapping outputs: the later one is written last, as the copies do
        same = out["phi"]
        a.fields(out={"phi": same, "rho": same, "ux": out["ux"], "uy": out["uy"], "p": out["p"]})
        assert np.array_equal(same, want["rho"])


def test_registered_memory(env):
    lbm, torch = env
    nx, ny = 320, 200
    with lbm.Lattice(nx, ny, **cases.params_static_drop()) as a:
        a.init(cases.drop(nx, ny, 50, 4.0)).step(3)
        want = a.fields()
        host = np.zeros((5, ny, nx))
        rt = torch.cuda.cudart()
        assert int(rt.cudaHostRegister(host.ctypes.data, host.nbytes, 0)) == 0
        try:
            a.fields(out=dict(zip(KEYS, host)))
        finally:
            rt.cudaHostUnregister(host.ctypes.data)
        for j, k in enumerate(KEYS):
            assert np.array_equal(host[j], want[k]), k
