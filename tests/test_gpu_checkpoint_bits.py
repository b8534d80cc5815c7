"""16-bit checkpoints, bit for bit: what is stored and restored against the same
roundings on the host.  The scale of a plane is the maximum over the shares of
eight CTAs (2048 groups of eight values per sweep); each plane here has its one large value
in another share, or in a second sweep, or none at all.  A scale of one share
only would keep the relative precision of BF16 and FP16, and no gate on a
gradient would see it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import paper_2007_06048_gb300 as M
from paper_2007_06048_gb300 import _build
from _gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "checkpoint_bits", "roundtrip.cu")
OUT = os.path.join(_build.ROOT, "_build", "checkpoint_bits")


@pytest.fixture(scope="module")
def lib():
    M.build()
    objs = [os.path.join(_build.OBJDIR, os.path.basename(s)[:-3] + ".o") for s in _build._sources()]
    if not all(os.path.exists(o) for o in objs):
        _build.build(force=True)
    os.makedirs(OUT, exist_ok=True)
    so = os.path.join(OUT, "libroundtrip.so")
    if not os.path.exists(so) or os.path.getmtime(so) < max(os.path.getmtime(p) for p in [SRC, *objs]):
        obj = os.path.join(OUT, "roundtrip.o")
        subprocess.run([_build.nvcc(), *_build.NVCC_FLAGS, "-c", SRC, "-o", obj], check=True)
        others = [o for o in objs if not o.endswith("mmod_adjoint.o")]
        subprocess.run([_build.nvcc(), *_build.ARCH, "-shared", "-cudart", "static", "-Xlinker", "-Bsymbolic", "-o", so,
                        obj, *others], check=True)
    lib = ctypes.CDLL(so)
    lib.roundtrip.argtypes = [ctypes.c_int] * 4 + [ctypes.c_void_p] * 7
    return lib


def _volume(nxp, ny, seed):
    """Planes 0 .. 7: the large value in the share of CTA 0 .. 7; 8: in its second sweep; 9: the last
    value; 10: zeros; 11: subnormals; 12: no large value."""
    rng = np.random.default_rng(seed)
    plane = nxp * ny
    u = (1e-3 * rng.standard_normal((13, plane))).astype(np.float32)
    for k in range(9):
        u[k, (8 * 256 * k + 8 * int(rng.integers(0, 256)) + int(rng.integers(0, 8))) % plane] = -37.0 - k
    u[9, -1] = 41.0
    u[10] = 0.0
    u[11] = (1e-41 * rng.standard_normal(plane)).astype(np.float32)
    return u


def _expected(u, dtype):
    import torch
    one, big = np.float32(1), np.float32(32767)
    if dtype == M.CKPT_BFP16:
        b = u.reshape(-1, 32)
        s = np.maximum(np.abs(b).max(1, keepdims=True), 32768 * np.finfo(np.float32).tiny)
        q = np.clip(np.rint(b * (big / s)), -32767, 32767).astype(np.int16)
        v = q.astype(np.float32) * (s / big)
        # half a step of the scale, and the roundings of the scale and of the product
        assert (np.abs(v - b.astype(np.float64)) <= s / 65534 * (1 + 2.0 ** -7)).all()
        return q.reshape(u.shape), s.ravel(), v.reshape(u.shape)
    s = np.maximum(np.abs(u).max(1, keepdims=True), np.finfo(np.float32).tiny)
    t = torch.from_numpy(u * (one / s)).to(torch.bfloat16 if dtype == M.CKPT_BF16 else torch.float16)
    return t.view(torch.int16).numpy(), s.ravel(), t.float().numpy() * s


@pytest.mark.parametrize("dtype", [M.CKPT_BF16, M.CKPT_FP16, M.CKPT_BFP16])
@pytest.mark.parametrize("nxp,ny", [(160, 130), (32, 9), (64, 1)])
def test_stored_and_restored_bits(lib, nxp, ny, dtype):
    torch = torch_cuda()
    u = [_volume(nxp, ny, seed) for seed in (1, 2)]
    nz = len(u[0])
    scales = nz if dtype != M.CKPT_BFP16 else u[0].size // 32
    dev = [torch.from_numpy(x).cuda() for x in u]
    out = [torch.full(u[0].shape, float("nan"), device="cuda") for _ in u]
    stored = torch.zeros((2, u[0].size), dtype=torch.int16, device="cuda")
    sc = torch.zeros((2, scales), device="cuda")
    torch.cuda.synchronize()
    err = lib.roundtrip(dtype, nxp, ny, nz, *(t.data_ptr() for t in (*dev, *out, stored, sc)), None)
    assert err == 0
    torch.cuda.synchronize()
    for i in range(2):
        q, s, v = _expected(u[i], dtype)
        assert np.array_equal(sc[i].cpu().numpy(), s)
        assert np.array_equal(stored[i].cpu().numpy(), q.ravel())
        assert np.array_equal(out[i].cpu().numpy().view(np.int32), v.view(np.int32))
