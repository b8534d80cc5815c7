"""Long source lists of the staggered system: one group per thread past warp 0
is looked up ahead, the rest after the plane loop, and lists of more than 1024
points go to the separate kernel: around each of those counts, with several
sources on one point, the plain kernels' bits."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from test_gpu_vd import run_vd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsrc", [1, 207, 208, 209, 225, 470, 1030])
@pytest.mark.parametrize("cpml", [False, True])
def test_source_counts_bitwise(nsrc, cpml):
    p = W.tiny_problem_vd(shape=(14, 37, 70), nt=20, nbl=4, nsrc=nsrc, nrec=50, seed=nsrc)
    p.cpml, p.cpml_f0 = cpml, 15.0
    if nsrc > 10:
        p.src_ijk[7] = p.src_ijk[3]
        p.src_ijk[nsrc - 1] = p.src_ijk[3]
    tr_t, st_t, prop = run_vd(p)
    assert prop.uses_tma and np.abs(st_t).max() > 0
    tr_s, st_s, _ = run_vd(p, kernel=M.KERNEL_SIMPLE)
    assert np.array_equal(tr_t, tr_s) and np.array_equal(st_t, st_s)
