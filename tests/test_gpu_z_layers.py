"""Groups of planes inside and outside the z layers run different code: layers that
meet (nz = 2 nbl), that end inside a group of four planes, that fill a z range or
leave it empty, with and without the free surface (no top layer), against the
plain kernel, bit for bit; z ranges forced to 5 and 8 planes shift the groups."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("zlen", [0, 5, 8])
@pytest.mark.parametrize("surface", [False, True])
@pytest.mark.parametrize("nz,nbl", [(8, 4), (9, 4), (12, 6), (13, 1), (26, 7), (41, 9), (33, 0)])
def test_z_layers_bitwise(nz, nbl, surface, zlen):
    p = W.tiny_problem(shape=(nz, 38, 75), nt=15, nbl=nbl, nsrc=4, nrec=100, seed=nz + nbl)
    p.free_surface = surface
    p.src_ijk[0] = [37, 19, nz - 1]
    p.src_ijk[1] = [20, 30, 1]
    tr_s, u_s, _ = run_gpu(p, kernel=M.KERNEL_SIMPLE)
    tr, u, _ = run_gpu(p, kernel=M.KERNEL_TMA, options={M.OPT_ZLEN: zlen} if zlen else None)
    assert np.abs(u).max() > 0
    assert np.array_equal(u, u_s) and np.array_equal(tr, tr_s)
