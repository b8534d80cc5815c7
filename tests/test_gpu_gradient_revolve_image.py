"""The binomial schedule's one-pass imaging term (A += psi (L u + s) inside a
step-shaped kernel) against the plain kernels, which write g and image in two
launches: bit for bit, for every compiled tile shape, with sources on top of
one another, on receivers, on tile corners and next to the surface; and the
two-launch form that longer source tables keep."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def gradient(p, resid, ckpt, kernel, variant=-1, dtype=M.CKPT_FP32):
    torch = torch_cuda()
    prop = M.Propagator.from_problem(p)
    prop.set_kernel(kernel)
    prop.set_variant(variant)
    prop.set_option(M.OPT_CKPT_SCHEME, M.SCHEME_REVOLVE)
    prop.set_model(torch.from_numpy(p.vel).cuda())
    g = torch.empty(p.vel.shape, device="cuda")
    prop.gradient(torch.from_numpy(p.wavelet).cuda(), torch.from_numpy(resid).cuda(), g, ckpt, dtype)
    return g.cpu().numpy()


@pytest.mark.parametrize("surface", [False, True])
@pytest.mark.parametrize("nsrc", [0, 1, 9, 240, 241])
@pytest.mark.parametrize("shape,nt", [((13, 25, 67), 9), ((6, 49, 41), 1), ((34, 33, 33), 4)])
def test_one_pass_imaging_bitwise(shape, nt, nsrc, surface):
    nz, ny, nx = shape
    p = W.tiny_problem(shape=shape, nt=nt, nbl=2, nsrc=nsrc, nrec=30, seed=nsrc + nz)
    p.free_surface = surface
    for s, q in enumerate([[nx - 1, ny - 1, nz - 1], [min(40, nx - 1), min(24, ny - 1), 1], [min(32, nx - 1), 16, 1]]):
        if s < nsrc:
            p.src_ijk[s] = q
    if nsrc > 5:
        p.src_ijk[4] = p.src_ijk[3]              # two sources on one point
        p.rec_ijk[0] = p.src_ijk[3]              # and a receiver
    resid = np.random.default_rng(4).standard_normal((nt, 30)).astype(np.float32)
    ref = gradient(p, resid, 3, M.KERNEL_SIMPLE)
    for v in (-1, 1, 2, *range(9, M.mmod_tma_variant_count())):
        assert np.array_equal(gradient(p, resid, 3, M.KERNEL_TMA, v), ref), v
