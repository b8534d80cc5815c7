"""CPML of the staggered system where a thread's memory variables are carried
from plane to plane: z ranges of one to a few planes, layers that end inside a
column pair, a row pair or next to a tile edge, layers that meet in the middle.
The TMA kernels must give the plain kernels' bits."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from test_gpu_vd import run_vd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("surface", [False, True])
@pytest.mark.parametrize("zlen", [None, 1, 3, 7])
@pytest.mark.parametrize("shape,nbl", [((24, 17, 65), 5), ((15, 32, 63), 7), ((21, 31, 128), 3), ((14, 14, 14), 7)])
def test_memory_variables_bitwise(shape, nbl, zlen, surface):
    p = W.tiny_problem_vd(shape=shape, nt=40, nbl=nbl, nsrc=3, nrec=9, seed=sum(shape))
    p.cpml, p.cpml_f0, p.free_surface = True, 15.0, surface
    tr_t, st_t, prop = run_vd(p, zlen=zlen)
    assert prop.uses_tma
    tr_s, st_s, _ = run_vd(p, kernel=M.KERNEL_SIMPLE)
    assert np.array_equal(tr_t, tr_s) and np.array_equal(st_t, st_s)
