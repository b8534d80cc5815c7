"""Traces of one handle on the device and on the host in turn, the device buffer
freed in between, so that the staging buffer of host traces may get its
address: the same bits every time."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cpml", [False, True])
def test_device_then_host_traces(cpml):
    torch = torch_cuda()
    p = W.tiny_problem(shape=(80, 90, 100), nt=120, nbl=8, nsrc=2, nrec=6000, seed=5)
    p.cpml, p.cpml_f0 = cpml, 15.0 if cpml else 0.0
    wav = torch.from_numpy(p.wavelet).cuda()
    ref = None
    for _ in range(3):
        prop = M.Propagator.from_problem(p)
        prop.set_model(torch.from_numpy(p.vel).cuda())
        dev = torch.empty((p.nt, len(p.rec_ijk)), device="cuda")
        prop.forward(wav, dev)
        got = dev.cpu().numpy()
        ref = got if ref is None else ref
        del dev
        torch.cuda.empty_cache()
        host = np.full(ref.shape, np.nan, np.float32)
        prop.forward(wav, host)
        assert np.abs(ref).max() > 0 and np.array_equal(got, ref) and np.array_equal(host, ref)
        prop.close()
