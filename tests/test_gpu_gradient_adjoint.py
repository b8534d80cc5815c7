"""mmod_gradient_adjoint: the velocity gradient and the adjoint sources from one
adjoint sweep are the bits of mmod_gradient and mmod_adjoint, for both
checkpoint schemes, every state kept, runs of one step, the plain kernels and
outputs in host memory."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [M.KERNEL_SIMPLE, M.KERNEL_TMA])
@pytest.mark.parametrize("nt,ckpt,scheme", [(1, 1, 0), (9, 3, 0), (10, 10, 0), (11, 3, 1)])
@pytest.mark.parametrize("surface", [False, True])
def test_gradient_adjoint_is_both_calls(nt, ckpt, scheme, kernel, surface):
    torch = torch_cuda()
    p = W.tiny_problem(shape=(13, 21, 45), nt=nt, nbl=2, nsrc=3, nrec=40, seed=79)
    p.free_surface = surface
    p.rec_ijk[0] = p.src_ijk[0]
    resid = np.random.default_rng(4).standard_normal((nt, 40)).astype(np.float32)
    prop = M.Propagator.from_problem(p)
    prop.set_kernel(kernel)
    prop.set_option(M.OPT_CKPT_SCHEME, scheme)
    prop.set_model(torch.from_numpy(p.vel).cuda())
    wav, res = torch.from_numpy(p.wavelet).cuda(), torch.from_numpy(resid).cuda()
    g, g2 = torch.empty(p.vel.shape, device="cuda"), torch.empty(p.vel.shape, device="cuda")
    a, a2 = torch.empty((3, nt), device="cuda"), np.full((3, nt), 7.0, np.float32)
    prop.gradient(wav, res, g, ckpt)
    prop.adjoint(res, a)
    prop.gradient_adjoint(wav, res, g2, a2, ckpt)
    assert torch.equal(g, g2) and np.array_equal(a.cpu().numpy(), a2)


def test_gradient_adjoint_needs_its_output():
    torch = torch_cuda()
    p = W.tiny_problem(shape=(13, 21, 45), nt=4, nbl=2, nsrc=1, nrec=4, seed=79)
    prop = M.Propagator.from_problem(p)
    prop.set_model(torch.from_numpy(p.vel).cuda())
    g = torch.empty(p.vel.shape, device="cuda")
    with pytest.raises(M.MmodError):
        prop.gradient_adjoint(torch.from_numpy(p.wavelet).cuda(), torch.zeros((4, 4), device="cuda"), g, None, 2)
