"""The box sizes the Poisson solver refuses: more than 65535 tiles of 8 rows (16 where the caller asks
for 16), whichever kernel and tile height it would choose, and more than 65535 segments."""
import ctypes as C

import pytest
import torch

from paper_2411_14631_gb300 import abi

pytestmark = pytest.mark.skipif(torch.cuda.is_available(), reason="fake device pointers: no-GPU check only")

FAKE = C.c_void_p(1 << 20)
ROWS = 65535 * 8


@pytest.mark.parametrize("nx,ny,nz,precond,tile_y,seg,refused",
                         [(1, ROWS, 9, 1, 0, 0, False), (1, ROWS + 1, 9, 1, 0, 0, True), (1, ROWS + 1, 9, 1, 16, 0, False),
                          (1, ROWS + 1, 9, 1, 8, 0, True), (1, 2 * ROWS + 1, 9, 1, 16, 0, True),
                          (1, ROWS + 1, 1, 0, 0, 0, True), (1, ROWS + 1, 9, 1, 0, 9, True),
                          (3, 4, 65536 * 4, 1, 0, 4, True), (3, 4, 65535 * 4, 1, 0, 4, False)])
def test_refused_sizes(nx, ny, nz, precond, tile_y, seg, refused):
    from paper_2411_14631_gb300 import build
    build.build()
    L = abi.lib()
    prm = abi.PpcgParams(nx, ny, nz, precond, 1e-4, 10, 0, tile_y, seg)
    nb = L.ppcg_workspace_bytes(nx, ny, nz)
    assert nb > 0
    # no iterations: a size that is accepted launches nothing
    st = L.ppcg_iterate(C.byref(prm), FAKE, FAKE, nb, None, 0, None)
    assert (st == abi.EINVAL) == refused, st
