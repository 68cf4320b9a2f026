"""lbm_create where no CUDA device can be used (child processes that see none):
LBM_ERR_CUDA for every size, storage format and boundary, from the planners'
smallest grids up.  The child must exit by itself: a signal fails the test."""
import os
import subprocess
import sys

import pytest

from paper_1710_09541_gb300 import build as lbm_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys
sys.path.insert(0, {root!r})
from paper_1710_09541_gb300 import lbm
for storage in (0, 1, 2, 3):
    for bc in (0, 1, 2):
        for kernel in (0, 1):
            try:
                lbm.Lattice({nx}, {ny}, storage=storage, bc_y=bc, kernel=kernel)
            except lbm.LbmError as e:
                assert e.status == lbm.LBM_ERR_CUDA, e
            else:
                raise AssertionError("created without a device")
"""


@pytest.mark.parametrize("nx,ny", [(2, 2), (8, 256), (64, 64), (200, 200), (501, 501), (2048, 2048)])
def test_create_without_a_device_returns_its_error(nx, ny):
    lbm_build.build()
    r = subprocess.run([sys.executable, "-c", CODE.format(root=ROOT, nx=nx, ny=ny)], capture_output=True, text=True,
                       env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0, (r.returncode, r.stderr)
