"""Tile shapes of the staged step kernel: every compiled variant (its tiles, tensor
maps and injection tables) against the plain kernel, bit for bit, on grids
around the edges of each shape; sources and receivers on tile corners; the
adjoint, whose injection points fill a plane; a variant changed between runs
of one handle; and the choice of variant with the options that need the
64 x 16 form."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import run_gpu, torch_cuda

pytestmark = pytest.mark.gpu


def _problem(shape, nt=20):
    nz, ny, nx = shape
    p = W.tiny_problem(shape=shape, nt=nt, nbl=min(3, min(shape) // 2), nsrc=6, nrec=nx * ny, seed=nx + ny + nz)
    edges = [(x, y) for x in (0, 31, 39, 40, 47, 48, 63, 64) for y in (0, 15, 16, 19, 20, 23, 24) if x < nx and y < ny]
    for s, (x, y) in enumerate(edges[-len(p.src_ijk):]):
        p.src_ijk[s] = [x, y, nz // 2]
    j, i = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    p.rec_ijk = np.stack([i.ravel(), j.ravel(), np.full(i.size, min(1, nz - 1))], 1).astype(np.int32)
    return p


def _adjoint(p, variant, kernel):
    torch = torch_cuda()
    prop = M.Propagator.from_problem(p)
    prop.set_kernel(kernel)
    prop.set_variant(variant)
    prop.set_model(torch.from_numpy(p.vel).cuda())
    resid = np.random.default_rng(5).standard_normal((p.nt, len(p.rec_ijk))).astype(np.float32)
    out = torch.empty((len(p.src_ijk), p.nt), device="cuda")
    prop.adjoint(torch.from_numpy(resid).cuda(), out)
    return out.cpu().numpy()


@pytest.mark.parametrize("variant", range(9, M.mmod_tma_variant_count()))
@pytest.mark.parametrize("shape", [(11, 21, 49), (14, 24, 40), (9, 33, 32), (10, 19, 95), (7, 49, 81), (6, 5, 3)])
def test_shapes_bitwise(shape, variant):
    p = _problem(shape)
    tr_s, u_s, _ = run_gpu(p, kernel=M.KERNEL_SIMPLE)
    tr, u, prop = run_gpu(p, kernel=M.KERNEL_TMA, variant=variant)
    assert prop.plan()["variant"] == variant
    assert np.array_equal(u, u_s) and np.array_equal(tr, tr_s)
    assert np.array_equal(_adjoint(p, variant, M.KERNEL_TMA), _adjoint(p, variant, M.KERNEL_SIMPLE))


def test_variants_in_turn_on_one_handle():
    torch = torch_cuda()
    p = _problem((12, 50, 90), nt=30)
    prop = M.Propagator.from_problem(p)
    prop.set_model(torch.from_numpy(p.vel).cuda())
    wav = torch.from_numpy(p.wavelet).cuda()
    resid = torch.from_numpy(np.random.default_rng(1).standard_normal((p.nt, len(p.rec_ijk))).astype(np.float32)).cuda()
    ref = None
    for v in [-1, *range(M.mmod_tma_variant_count()), -1]:
        prop.set_variant(v)
        tr = torch.empty((p.nt, len(p.rec_ijk)), device="cuda")
        g = torch.empty(p.vel.shape, device="cuda")
        prop.forward(wav, tr)
        prop.gradient(wav, resid, g, 4)
        got = tr.cpu().numpy(), g.cpu().numpy()
        ref = ref or got
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]), v


def test_options_keep_their_forms():
    torch = torch_cuda()
    p = _problem((40, 50, 90), nt=10)
    prop = M.Propagator.from_problem(p)
    prop.set_model(torch.from_numpy(p.vel).cuda())
    auto = prop.plan()["variant"]
    prop.set_option(M.OPT_PERSISTENT, 1)
    assert prop.plan()["variant"] == 2 and prop.persistent_grid() > 0
    prop.set_option(M.OPT_PERSISTENT, 0)
    prop.set_option(M.OPT_CLAIM, 8)
    assert prop.plan()["variant"] == 2 and prop.plan()["planes_per_chunk"] == 8
    prop.set_option(M.OPT_CLAIM, 0)
    assert prop.plan()["variant"] == auto
    with pytest.raises(M.MmodError):
        M.Batch([prop]).set_variant(9)
