"""Tile shapes of the staggered kernels: grids for which the plan takes each of
them, ragged by a few cells, damping and CPML, with and without a free surface:
the plain kernels' bits."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from test_gpu_vd import run_vd

pytestmark = pytest.mark.gpu

# (nz, ny, nx) and the (width, height) of the tiles the plan takes there
GRIDS = [((14, 16, 64), (64, 16)), ((46, 57, 72), (48, 20)), ((37, 70, 72), (40, 24)), ((43, 62, 90), (32, 32)),
         ((43, 88, 90), (64, 16))]   # equal planes and counts in 40 x 24: stays 64 x 16


@pytest.mark.parametrize("surface", [False, True])
@pytest.mark.parametrize("cpml", [False, True])
@pytest.mark.parametrize("shape,tile", GRIDS)
def test_tile_shapes_bitwise(shape, tile, cpml, surface):
    p = W.tiny_problem_vd(shape=shape, nt=25, nbl=6, nsrc=5, nrec=200, seed=sum(shape))
    p.cpml, p.cpml_f0, p.free_surface = cpml, 15.0, surface
    nz, ny, nx = shape
    p.src_ijk[0] = [min(tile[0], nx - 1), min(tile[1], ny - 1), nz // 2]
    p.src_ijk[1] = [nx - 1, ny - 1, nz - 1]
    tr_t, st_t, prop = run_vd(p)
    plan = prop.plan()
    assert prop.uses_tma and (plan["tiles_x"], plan["tiles_y"]) == (-(-nx // tile[0]), -(-ny // tile[1]))
    tr_s, st_s, _ = run_vd(p, kernel=M.KERNEL_SIMPLE)
    assert np.array_equal(tr_t, tr_s) and np.array_equal(st_t, st_s)
