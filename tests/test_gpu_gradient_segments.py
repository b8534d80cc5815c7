"""Segments with FP32 checkpoints, whose states stay where the first sweep's
steps left them: every segment length down to two, odd and even, with and
without a shorter last segment, against the binomial schedule (which copies
its states) and the plain kernels, bit for bit."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def gradient(p, resid, ckpt, scheme=M.SCHEME_SEGMENTS, kernel=M.KERNEL_AUTO, prop=None):
    torch = torch_cuda()
    prop = prop or M.Propagator.from_problem(p)
    prop.set_kernel(kernel)
    prop.set_option(M.OPT_CKPT_SCHEME, scheme)
    prop.set_model(torch.from_numpy(p.vel).cuda())
    g = torch.empty(p.vel.shape, device="cuda")
    prop.gradient(torch.from_numpy(p.wavelet).cuda(), torch.from_numpy(resid).cuda(), g, ckpt)
    return g.cpu().numpy()


@pytest.mark.parametrize("surface", [False, True])
@pytest.mark.parametrize("nt", [2, 3, 8, 13])
def test_segment_lengths_bitwise(nt, surface):
    p = W.tiny_problem(shape=(13, 21, 45), nt=nt, nbl=2, nsrc=3, nrec=40, seed=79)
    p.free_surface = surface
    p.rec_ijk[0] = p.src_ijk[0]
    resid = np.random.default_rng(4).standard_normal((nt, 40)).astype(np.float32)
    ref = gradient(p, resid, 2, M.SCHEME_REVOLVE)
    prop = M.Propagator.from_problem(p)   # one handle: layouts of different slot counts in turn
    for ckpt in range(1, nt + 1):
        assert np.array_equal(gradient(p, resid, ckpt, prop=prop), ref), ckpt
        assert np.array_equal(gradient(p, resid, ckpt, kernel=M.KERNEL_SIMPLE), ref), ckpt
