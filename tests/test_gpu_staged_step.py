"""The staged step kernel at the lengths and edges where its schedule changes:
z ranges of one to nine planes (one group of four planes, its remainders, both
halves of the halo ring), grids a few cells around a tile's edge, with and
without the free surface's image planes.  Bit for bit the plain kernel's
wavefield and traces."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("surface", [False, True])
@pytest.mark.parametrize("zlen", [0, 1, 2, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("shape", [(19, 17, 65), (9, 33, 48), (13, 16, 127), (5, 1, 1), (22, 41, 81)])
def test_plane_ranges_bitwise(shape, zlen, surface):
    p = W.tiny_problem(shape=shape, nt=25, nbl=min(3, min(shape) // 2), nsrc=4, nrec=12, seed=sum(shape))
    p.free_surface = surface
    tr_s, u_s, _ = run_gpu(p, kernel=M.KERNEL_SIMPLE)
    tr, u, _ = run_gpu(p, kernel=M.KERNEL_TMA, options={M.OPT_ZLEN: zlen})
    assert np.array_equal(u, u_s) and np.array_equal(tr, tr_s)
