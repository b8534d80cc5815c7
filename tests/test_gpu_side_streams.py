"""Handles used on a non-blocking stream while the default stream is busy: a run
may rely on nothing that the default stream still has to do.  Tile shapes
selected by variant, option and batch mode right before the run; the same bits as
on the default stream."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

CHANGES = [None, ("variant", 2), ("variant", 10), ("option", M.OPT_PERSISTENT, 1), ("option", M.OPT_CLAIM, 8)]


def _problem(seed=9):
    return W.tiny_problem(shape=(40, 100, 130), nt=40, nbl=8, nsrc=4, nrec=5000, seed=seed)


def _run(p, stream, change):
    torch = torch_cuda()
    vel, wav = torch.from_numpy(p.vel).cuda(), torch.from_numpy(p.wavelet).cuda()
    resid = torch.from_numpy(np.random.default_rng(1).standard_normal((p.nt, 5000)).astype(np.float32)).cuda()
    tr, adj, g = (torch.empty(s, device="cuda") for s in ((p.nt, 5000), (4, p.nt), p.vel.shape))
    torch.cuda.synchronize()
    if stream is not None:
        torch.cuda._sleep(40_000_000)   # some 20 ms of work on the default stream
    s = None if stream is None else stream.cuda_stream
    prop = M.Propagator.from_problem(p)
    prop.set_model(vel, s)
    if change:
        prop.set_variant(change[1]) if change[0] == "variant" else prop.set_option(*change[1:])
    prop.forward(wav, tr, None, s)
    prop.adjoint(resid, adj, s)
    prop.gradient(wav, resid, g, 4, M.CKPT_FP32, s)
    torch.cuda.synchronize()
    prop.close()
    return [t.cpu().numpy() for t in (tr, adj, g)]


@pytest.mark.parametrize("change", CHANGES)
def test_side_stream_bitwise(change):
    torch = torch_cuda()
    p = _problem()
    ref = _run(p, None, None)
    got = _run(p, torch.cuda.Stream(), change)
    for a, b in zip(got, ref):
        assert np.abs(b).max() > 0 and np.array_equal(a, b)


@pytest.mark.parametrize("mode", [M.BATCH_STREAMS, M.BATCH_FUSED, M.BATCH_PERSISTENT])
def test_batch_on_a_side_stream_bitwise(mode):
    torch = torch_cuda()
    shots = [_problem(seed) for seed in (9, 10, 11)]
    vel = [torch.from_numpy(p.vel).cuda() for p in shots]
    wav = [torch.from_numpy(p.wavelet).cuda() for p in shots]
    tr = [torch.empty((p.nt, 5000), device="cuda") for p in shots]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(40_000_000)
    props = [M.Propagator.from_problem(p) for p in shots]
    for prop, v in zip(props, vel):
        prop.set_model(v, s.cuda_stream)
    b = M.Batch(props)
    b.set_mode(mode)
    b.forward(wav, tr, s.cuda_stream)
    torch.cuda.synchronize()
    b.close()
    for p, t in zip(shots, tr):
        ref = _run(p, None, None)[0]
        assert np.abs(ref).max() > 0 and np.array_equal(t.cpu().numpy(), ref)


@pytest.mark.parametrize("cpml", [False, True])
def test_staggered_on_a_side_stream_bitwise(cpml):
    torch = torch_cuda()
    p = W.tiny_problem_vd(shape=(40, 100, 130), nt=40, nbl=8, nsrc=4, nrec=5000, seed=9)
    p.cpml, p.cpml_f0 = cpml, 15.0 if cpml else 0.0
    out = []
    for stream in (None, torch.cuda.Stream()):
        vel, rho, wav = (torch.from_numpy(a).cuda() for a in (p.vel, p.rho, p.wavelet))
        tr = torch.empty((p.nt, 5000), device="cuda")
        torch.cuda.synchronize()
        s = None
        if stream is not None:
            s = stream.cuda_stream
            torch.cuda._sleep(40_000_000)
        prop = M.StaggeredPropagator.from_problem(p)
        prop.set_model(vel, rho, s)
        prop.forward(wav, tr, stream=s)
        torch.cuda.synchronize()
        prop.close()
        out.append(tr.cpu().numpy())
    assert np.abs(out[0]).max() > 0 and np.array_equal(out[0], out[1])
