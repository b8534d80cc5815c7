"""Gradients with 16-bit checkpoints, programmatic dependent launch off and on:
the same bits.  Several waves of CTAs per step (z ranges of four planes), so that
a step's first CTAs start while others of the kernel in front still run, and
segments of two and three steps, so that every few steps follow a restore."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [M.CKPT_FP32, M.CKPT_BF16, M.CKPT_FP16, M.CKPT_BFP16])
@pytest.mark.parametrize("scheme,ckpt", [(M.SCHEME_SEGMENTS, 6), (M.SCHEME_SEGMENTS, 4), (M.SCHEME_REVOLVE, 3)])
def test_pdl_keeps_the_bits(scheme, ckpt, dtype):
    torch = torch_cuda()
    p = W.tiny_problem(shape=(48, 230, 260), nt=12, nbl=8, nsrc=3, nrec=50, seed=31)
    p.rec_ijk[:] = np.clip(p.src_ijk[np.arange(50) % 3] + np.random.default_rng(1).integers(-4, 5, (50, 3)), 0,
                           np.array([260, 230, 48]) - 1)
    resid = torch.from_numpy(np.random.default_rng(2).standard_normal((p.nt, 50)).astype(np.float32)).cuda()
    wav = torch.from_numpy(p.wavelet).cuda()
    out = []
    for pdl in (0, 1, 1):
        prop = M.Propagator.from_problem(p)
        prop.set_option(M.OPT_PDL, pdl)
        prop.set_option(M.OPT_ZLEN, 4)
        prop.set_option(M.OPT_CKPT_SCHEME, scheme)
        prop.set_model(torch.from_numpy(p.vel).cuda())
        for _ in range(2):   # a first pass and one on the kept work space
            g = torch.empty(p.vel.shape, device="cuda")
            prop.gradient(wav, resid, g, ckpt, dtype)
            out.append(g.cpu().numpy())
        assert prop.plan()["grid"] > 2 * 304
        prop.close()
    assert np.abs(out[0]).max() > 0
    for g in out[1:]:
        assert np.array_equal(g, out[0])
