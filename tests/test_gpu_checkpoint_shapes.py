"""16-bit checkpoints on planes of very different sizes.

The compression of a plane is shared by a cluster of eight CTAs of 256 threads
with eight values per thread (16 384 values per sweep): planes far smaller (most
CTAs hold nothing), just above, and several sweeps long, ragged on x.  One
16-bit save and restore of every state against the FP32 gradient, with the
gates of the 30 Hz checkpoint cases (the storage error is the same per value).
"""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import rel_l2, torch_cuda

pytestmark = pytest.mark.gpu


def _gradient(p, resid, ckpt, dtype, scheme):
    torch = torch_cuda()
    prop = M.Propagator.from_problem(p)
    prop.set_option(M.OPT_CKPT_SCHEME, scheme)
    prop.set_model(torch.from_numpy(p.vel).cuda())
    g = torch.empty(p.vel.shape, device="cuda")
    prop.gradient(torch.from_numpy(p.wavelet).cuda(), torch.from_numpy(resid).cuda(), g, ckpt, dtype)
    return g.cpu().numpy()


@pytest.mark.parametrize("scheme", [M.SCHEME_SEGMENTS, M.SCHEME_REVOLVE])
@pytest.mark.parametrize("shape", [(40, 9, 33), (18, 130, 125), (12, 300, 257)])
@pytest.mark.parametrize("dtype,gate", [(M.CKPT_BF16, 2e-2), (M.CKPT_FP16, 3e-3), (M.CKPT_BFP16, 1e-3)])
def test_checkpoint_plane_sizes(shape, dtype, gate, scheme):
    p = W.tiny_problem(shape=shape, nt=40, nbl=4 if min(shape) > 8 else 2, nsrc=1, nrec=9, seed=21)
    # receivers a few cells from the source, so that the gradient is not zero on the wide planes
    i, j, k = p.src_ijk[0] = [shape[2] // 2, shape[1] // 2, shape[0] // 2]
    p.rec_ijk[:] = [[i - 4 + r, min(j + 2, shape[1] - 1), k - 2] for r in range(9)]
    resid = np.random.default_rng(3).standard_normal((p.nt, 9)).astype(np.float32)
    g32 = _gradient(p, resid, 5, M.CKPT_FP32, scheme)
    g16 = _gradient(p, resid, 5, dtype, scheme)
    assert np.isfinite(g16).all() and np.abs(g32).max() > 0
    assert rel_l2(g16, g32) <= gate
