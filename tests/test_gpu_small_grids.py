"""Grids that fit one CTA per SM: the z split chosen there (a CTA alone on its SM
takes 0.6 of the time per plane) and grids on both sides of that line, against
the plain kernel, bit for bit."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import run_gpu, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(64, 64, 64), (56, 56, 56), (72, 72, 72), (96, 96, 96), (37, 61, 50), (5, 17, 129),
                                   (150, 16, 64), (153, 15, 60)])
@pytest.mark.parametrize("surface", [False, True])
def test_small_grids_bitwise(shape, surface):
    torch = torch_cuda()
    p = W.tiny_problem(shape=shape, nt=12, nbl=2, nsrc=5, nrec=300, seed=sum(shape))
    p.free_surface = surface
    tr_s, u_s, _ = run_gpu(p, kernel=M.KERNEL_SIMPLE)
    tr, u, prop = run_gpu(p, kernel=M.KERNEL_TMA)
    assert np.array_equal(u, u_s) and np.array_equal(tr, tr_s)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if shape == (64, 64, 64) and sms >= 128:   # 4 tiles x 32 ranges of 2 planes, one CTA per SM
        assert prop.plan()["planes_per_chunk"] == 2
