"""The work a user of the propagator library has it do, as timed cases.

Every case is one call (or one training-style iteration) through the package's
public entry points on a model that a survey would bring: layered velocities
with a smooth perturbation, Ricker sources near the surface, receivers on a
plane, absorbing layers on the faces.  Grid sizes are those of this
repository's workloads, tests and benchmark, or generic odd ones; the number
of time steps is shortened so that a pass stays well under a second (every
step costs the same).

A case is a dict of plain values:
  kind      "forward", "adjoint", "gradient", "fwi" (autograd iteration),
            "vd" (staggered variable-density run), "batch" (uneven shots)
  nx ny nz  grid; nt time steps; nbl layer width; h spacing (m)
  nsrc      point sources at depth src_k; receivers on the plane rec_k with
            stride rec_stride on both axes
  surface   free surface at k = 0; cpml: CPML layers instead of damping ones
  optimised dispersion-optimised stencil weights instead of the Taylor ones
  ckpt, ckpt_dtype, revolve   checkpoints of the gradient
  shots, size_seed            batch only: the shots' sizes come from size_seed
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2007_06048_gb300 as M
from paper_2007_06048_gb300.autograd import forward_map

H = 10.0                       # grid spacing, m
V_LO, V_HI = 1500.0, 4500.0    # velocities of the layered models, m/s
V_TOP = 1.05 * V_HI            # bound of the perturbed model: fixes dt at CFL 0.4
DT = 0.4 * H / V_TOP
REFL = 1e-3
F0 = 2.0                       # CPML frequency shift, Hz


def _case(kind, nx, ny, nz, nt, nbl, **kw):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, nt=nt, nbl=nbl, nsrc=1, src_k=4, rec_k=0, rec_stride=1,
             surface=False, cpml=False, optimised=False)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call in use: a 64^3 model, a hundred steps, a handful of
        # receivers (tutorials, unit checks, parameter scans over tiny models).
        _case("forward", 64, 64, 64, 100, 8, src_k=8, rec_k=4, rec_stride=16, name="forward_small"),
        # A near-surface survey on an odd-sized box: free surface, three
        # sources, optimised weights for a coarse grid.
        _case("forward", 151, 117, 98, 300, 12, nsrc=3, surface=True, optimised=True, rec_k=1, rec_stride=3,
              name="forward_ragged_surface"),
        # The benchmark's shot: 240^3, 20-cell layers, a receiver at every surface point.
        _case("forward", 240, 240, 240, 300, 20, name="forward_240"),
        # One large shot, far beyond the caches.
        _case("forward", 1024, 1024, 512, 40, 32, name="forward_large"),
        # The transpose of the benchmark's shot: every surface point injects.
        _case("adjoint", 240, 240, 240, 300, 20, name="adjoint_240"),
        # Velocity gradient at the size of the inversion workload, FP32 checkpoints.
        _case("gradient", 200, 200, 200, 400, 20, rec_stride=3, ckpt=20, ckpt_dtype=0, revolve=False,
              name="gradient_200"),
        # Gradient of a smaller odd box under a tight memory budget: binomial
        # checkpointing with 16-bit storage.
        _case("gradient", 133, 144, 120, 200, 16, rec_stride=4, ckpt=10, ckpt_dtype=1, revolve=True,
              name="gradient_revolve_bf16"),
        # One full-waveform-inversion iteration through autograd: new model,
        # forward run, misfit, gradients in the velocity and the wavelet.
        _case("fwi", 160, 120, 100, 250, 16, nsrc=2, rec_k=2, rec_stride=4, ckpt=16, ckpt_dtype=0,
              name="fwi_iteration"),
        # The benchmark's shot with CPML layers.
        _case("forward", 240, 240, 240, 150, 20, cpml=True, name="cpml_240"),
        # The benchmark's shot in the variable-density staggered system.
        _case("vd", 240, 240, 240, 150, 20, name="vd_240"),
        # A variable-density survey on an odd box: CPML layers under a free surface.
        _case("vd", 176, 150, 123, 200, 12, nsrc=2, surface=True, cpml=True, rec_k=1, rec_stride=4,
              name="vd_cpml_surface"),
        # Several shots of uneven size advanced together (default mode).
        _case("batch", 0, 0, 0, 150, 20, rec_stride=4, shots=8, size_seed=4, name="batch_8"),
    ]


def draw(rng):
    """One more case of the same ranges (sizes log-uniform, odd ones among them)."""
    kind = rng.choice(["forward", "forward", "forward", "adjoint", "gradient", "fwi", "vd", "vd", "batch"])
    # upper bound of points x steps: what each kind does per step, against the
    # largest listed case
    budget = {"forward": 1.0e10, "adjoint": 1.0e10, "gradient": 2.0e9, "fwi": 1.5e9, "vd": 3.0e9}
    src_k, rec_k = rng.choice([2, 4, 8]), rng.choice([0, 1, 4])
    if kind == "batch":
        return _case("batch", 0, 0, 0, rng.choice([60, 90, 120]), rng.choice([12, 16, 20]), rec_stride=rng.choice([3, 4]),
                     shots=rng.randint(3, 8), size_seed=rng.randrange(1, 10 ** 6), src_k=src_k, rec_k=rec_k)
    nt = rng.choice([60, 100, 150, 200, 300])
    hi = 400.0 if kind in ("forward", "adjoint") else 240.0
    while True:
        nx, ny, nz = (int(round(math.exp(rng.uniform(math.log(40.0), math.log(hi))))) for _ in range(3))
        if nx * ny * nz * nt <= budget[kind]:
            break
    nbl = rng.choice([w for w in (8, 12, 16, 20, 32) if 2 * w + 12 <= min(nx, ny, nz)] or [8])
    c = _case(kind, nx, ny, nz, nt, nbl, nsrc=rng.choice([1, 1, 2, 5]), src_k=src_k, rec_k=rec_k,
              rec_stride=rng.choice([1, 2, 4]), surface=rng.random() < 0.3)
    if c["surface"]:
        c["rec_k"] = max(1, rec_k)   # the surface plane itself records zeros
    if kind in ("forward", "vd"):
        c["cpml"] = rng.random() < 0.35
    if kind == "forward" and not c["cpml"]:
        c["optimised"] = rng.random() < 0.25
    if kind == "gradient":
        c["ckpt"], c["ckpt_dtype"], c["revolve"] = rng.choice([8, 12, 20]), rng.choice([0, 0, 2, 3]), rng.random() < 0.4
    if kind == "fwi":
        c["ckpt"], c["ckpt_dtype"] = rng.choice([8, 16]), 0
    return c


# ---- inputs -----------------------------------------------------------------

def _device():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def _gen(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _smooth(shape, gen, cells=8):
    """Smooth random field in [-1, 1]: coarse noise interpolated to the grid."""
    coarse = torch.rand((1, 1) + tuple(max(2, n // cells + 1) for n in shape), generator=gen, device=_device()) * 2 - 1
    return torch.nn.functional.interpolate(coarse, size=shape, mode="trilinear", align_corners=True)[0, 0]


def _velocity(shape, seed):
    """Four flat layers, interfaces at random depths, times (1 + 5 % smooth field)."""
    nz = shape[0]
    rng = random.Random(seed)
    depths = sorted(rng.sample(range(nz // 6, nz - 2), 3))
    layers = np.array([1500.0, 2200.0, 3000.0, 4500.0], np.float32)
    vz = torch.from_numpy(layers[np.searchsorted(depths, np.arange(nz), side="right")]).to(_device())
    vel = _smooth(shape, _gen(seed + 1))
    return vel.mul_(0.0499).add_(1.0).mul_(vz[:, None, None]).contiguous()


def _density(vel, seed):
    """Gardner's rule on the velocity times (1 + 3 % smooth field)."""
    return (310.0 * vel ** 0.25 * (1.0 + 0.03 * _smooth(tuple(vel.shape), _gen(seed + 2)))).contiguous()


def _ricker(f, nt, shift=0.0):
    t = np.arange(nt, dtype=np.float64) * DT - 1.2 / f - shift
    a = (np.pi * f * t) ** 2
    return (1.0 - 2.0 * a) * np.exp(-a)


def _peak(nt):
    """Peak frequency whose wavelet is over within the run, at most 25 Hz on 10 m cells."""
    return max(12.0, min(25.0, 3.0 / (nt * DT)))


def _wavelets(case, seed):
    rng = random.Random(seed + 3)
    f = _peak(case["nt"])
    w = [rng.uniform(0.5, 2.0) * _ricker(f * rng.uniform(0.8, 1.2), case["nt"]) for _ in range(case["nsrc"])]
    return np.ascontiguousarray(np.stack(w), np.float32)


def _geometry(case, seed):
    """Sources at seeded places away from the sides, receivers on a plane."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = random.Random(seed + 5)
    src = [[rng.randint(nx // 3, 2 * nx // 3), rng.randint(ny // 3, 2 * ny // 3), min(case["src_k"], nz - 1)]
           for _ in range(case["nsrc"])]
    st = case["rec_stride"]
    j, i = np.meshgrid(np.arange(0, ny, st), np.arange(0, nx, st), indexing="ij")
    rec = np.stack([i.ravel(), j.ravel(), np.full(i.size, min(case["rec_k"], nz - 1))], 1)
    return np.array(src, np.int32), np.ascontiguousarray(rec, np.int32)


def _residual(case, nrec, seed):
    """Band-limited data [nt][nrec]: a Ricker pulse per receiver with its own amplitude and arrival."""
    nt, g = case["nt"], _gen(seed + 7)
    f = _peak(nt)
    t = torch.arange(nt, device=_device(), dtype=torch.float32)[:, None] * DT
    t0 = torch.rand((1, nrec), generator=g, device=_device()) * (nt * DT * 0.5) + 1.2 / f
    amp = torch.randn((1, nrec), generator=g, device=_device())
    a = (math.pi * f * (t - t0)) ** 2
    return (amp * (1.0 - 2.0 * a) * torch.exp(-a)).contiguous()


def _shots(case):
    """The batch's shots as forward cases: sizes from size_seed, in steps of 16 and odd ones."""
    rng = random.Random(case["size_seed"])
    out = []
    for s in range(case["shots"]):
        n = [rng.randrange(96, 257, 16) + (rng.randrange(0, 15) if rng.random() < 0.4 else 0) for _ in range(3)]
        out.append(_case("forward", n[0], n[1], n[2], case["nt"], case["nbl"], src_k=case["src_k"],
                         rec_k=case["rec_k"], rec_stride=case["rec_stride"]))
    return out


def _inputs(case, seed):
    """Everything drawn from the seed: velocity (device), sources, receivers, wavelets."""
    src, rec = _geometry(case, seed)
    vel = _velocity((case["nz"], case["ny"], case["nx"]), seed)
    return vel, src, rec, _wavelets(case, seed)


def _propagator(case, src, rec):
    shape = (case["nz"], case["ny"], case["nx"])
    p = M.Propagator(shape, (H, H, H), DT, case["nt"], nbl=case["nbl"], src_ijk=src, rec_ijk=rec, damp_R=REFL,
                     free_surface=case["surface"], cpml=case["cpml"], cpml_f0=F0 if case["cpml"] else 0.0)
    if case["optimised"]:
        p.set_fd_coefficients(M.mmod_optimized_coefficients(2.0 * math.pi / 3.0))
    return p


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        props, wavs, traces = [], [], []
        for s, c in enumerate(_shots(case)):
            vel, src, rec, wav = _inputs(c, seed + 100 * s)
            p = _propagator(c, src, rec)
            p.set_model(vel)
            props.append(p)
            wavs.append(torch.from_numpy(wav).cuda())
            traces.append(torch.empty((c["nt"], len(rec)), device="cuda"))
        return dict(kind=kind, batch=M.Batch(props), wavs=wavs, traces=traces)
    vel, src, rec, wav = _inputs(case, seed)
    st = dict(kind=kind, wav=torch.from_numpy(wav).cuda())
    shape = tuple(vel.shape)
    if kind == "vd":
        p = M.StaggeredPropagator(shape, (H, H, H), DT, case["nt"], nbl=case["nbl"], src_ijk=src, rec_ijk=rec,
                                  damp_R=REFL, cpml=case["cpml"], cpml_f0=F0 if case["cpml"] else 0.0,
                                  free_surface=case["surface"])
        p.set_model(vel, _density(vel, seed))
        st.update(prop=p, traces=torch.empty((case["nt"], len(rec)), device="cuda"),
                  final=torch.empty((4,) + shape, device="cuda"))
        return st
    p = _propagator(case, src, rec)
    st["prop"] = p
    if kind == "fwi":
        st.update(vel=vel.requires_grad_(), data=_residual(case, len(rec), seed), ckpt=(case["ckpt"], case["ckpt_dtype"]))
        st["wav"].requires_grad_()
        return st
    p.set_model(vel)
    if kind == "forward":
        st.update(traces=torch.empty((case["nt"], len(rec)), device="cuda"), final=torch.empty(shape, device="cuda"))
    elif kind == "adjoint":
        st.update(resid=_residual(case, len(rec), seed), out=torch.empty((case["nsrc"], case["nt"]), device="cuda"))
    elif kind == "gradient":
        if case["revolve"]:
            p.set_option(M.OPT_CKPT_SCHEME, M.SCHEME_REVOLVE)
        st.update(resid=_residual(case, len(rec), seed), out=torch.empty(shape, device="cuda"),
                  ckpt=(case["ckpt"], case["ckpt_dtype"]))
    return st


def run(st):
    kind = st["kind"]
    if kind == "batch":
        st["batch"].forward(st["wavs"], st["traces"])
        return st["traces"]
    p = st["prop"]
    if kind in ("forward", "vd"):
        p.forward(st["wav"], st["traces"], st["final"])
        return st["traces"], st["final"]
    if kind == "adjoint":
        p.adjoint(st["resid"], st["out"])
        return st["out"]
    if kind == "gradient":
        p.gradient(st["wav"], st["resid"], st["out"], *st["ckpt"])
        return st["out"]
    traces = forward_map(p, st["vel"], st["wav"], *st["ckpt"])
    misfit = 0.5 * ((traces - st["data"]) ** 2).sum()
    gv, gw = torch.autograd.grad(misfit, (st["vel"], st["wav"]))
    return traces.detach(), gv, gw


def work(case):
    """Bytes and operations of one pass.  A step cannot do without reading
    u^n, u^{n-1} and c and writing u^{n+1} (16 B per point; the staggered system
    reads p, v, K, b and writes p, v: 40 B); CPML layers add psi and zeta read
    and written (16 B) per cell and axis; the gradient is a forward, an
    adjoint and a product sweep (16 + 16 + 8 B, g^n written and read)."""
    if case["kind"] == "batch":
        parts = [work(c) for c in _shots(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nx, ny, nz, nt = case["nx"], case["ny"], case["nz"], case["nt"]
    pts = float(nx) * ny * nz
    nrec = -(-nx // case["rec_stride"]) * -(-ny // case["rec_stride"])
    traces = 4.0 * nrec * nt
    per = {"forward": 16.0, "adjoint": 16.0, "gradient": 40.0, "fwi": 16.0 + 40.0 + 16.0, "vd": 40.0}[case["kind"]]
    ops = {"forward": 44.0, "adjoint": 44.0, "gradient": 90.0, "fwi": 178.0, "vd": 80.0}[case["kind"]]
    total = per * pts * nt
    if case["cpml"]:
        faces = 2.0 / nx + 2.0 / ny + (1.0 if case["surface"] else 2.0) / nz
        # per layer cell and axis: 8 B read + 8 B written for each memory variable pair
        total += 16.0 * pts * case["nbl"] * faces * nt
        ops += 40.0 * case["nbl"] * faces
    fields = {"forward": 1, "adjoint": 0, "gradient": 1, "fwi": 1, "vd": 4}[case["kind"]]
    return {"bytes": total + traces + 4.0 * fields * pts, "flops": ops * pts * nt}


# ---- 64-bit reference -------------------------------------------------------

R = 4
TAYLOR = (8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)
FIRST = (4.0 / 5.0, -1.0 / 5.0, 4.0 / 105.0, -1.0 / 280.0)              # centred first difference
STAGGERED = (1225.0 / 1024.0, -245.0 / 3072.0, 49.0 / 5120.0, -5.0 / 7168.0)


def _optimised_weights(kmax):
    """c_m minimising the integral over [0, kmax] of (2 sum c_m (1 - cos m k) / k^2 - 1)^2 with sum m^2 c_m = 1."""
    x, w = np.polynomial.legendre.leggauss(200)
    k, w = 0.5 * kmax * (x + 1.0), 0.5 * kmax * w
    m = np.arange(1, R + 1)
    b = 2.0 * (1.0 - np.cos(np.outer(k, m))) / k[:, None] ** 2
    a = np.zeros((R + 1, R + 1))
    rhs = np.zeros(R + 1)
    a[:R, :R] = (b * w[:, None]).T @ b
    a[:R, R] = a[R, :R] = m ** 2
    rhs[:R], rhs[R] = b.T @ w, 1.0
    return tuple(np.linalg.solve(a, rhs)[:R])


def _sh(u, axis, m):
    """The padded array u [nz+8][ny+8][nx+8] shifted by m along axis (0 z, 1 y, 2 x), interior extent."""
    s = [slice(R, -R)] * 3
    s[axis] = slice(R + m, u.shape[axis] - R + m)
    return u[tuple(s)]


def _padded(shape, dev):
    return torch.zeros([n + 2 * R for n in shape], dtype=torch.float64, device=dev)


def _odd_image(u):
    for m in range(1, R + 1):
        u[R - m] = -u[R + m]


class _Ref:
    """Model, layers and stepping of the second-order equation in 64 bits."""

    def __init__(self, case, vel):
        self.case, self.dev, self.shape = case, vel.device, tuple(vel.shape)
        self.vel = vel.double()
        self.vmax = float(self.vel.max())
        self.C = (DT * DT) * self.vel * self.vel
        nbl, n3 = case["nbl"], self.shape
        self.tmp = torch.empty(self.shape, dtype=torch.float64, device=self.dev)
        self.L = torch.empty_like(self.tmp)
        self.w = [x / (H * H) for x in (_optimised_weights(2.0 * math.pi / 3.0) if case["optimised"] else TAYLOR)]
        prof = []
        for a in range(3):
            d = self.depth(a, np.arange(n3[a], dtype=np.float64))
            eta = 3.0 * self.vmax * math.log(1.0 / REFL) / (2.0 * nbl * H) * (d / nbl) ** 2 * DT
            prof.append(torch.from_numpy(eta).to(self.dev))
        self.e = prof[0][:, None, None] + prof[1][None, :, None] + prof[2][None, None, :]

    def depth(self, a, x):
        """Cells into the layers of axis a (0 z, 1 y, 2 x) at positions x; no layer under a free surface."""
        n, nbl = self.shape[a], self.case["nbl"]
        d = np.maximum(x - (n - 1 - nbl), 0.0)
        if not (a == 0 and self.case["surface"]):
            d = np.maximum(d, nbl - x)
        return np.minimum(d, nbl)

    def axis_term(self, u, a, out):
        out.zero_()
        c = _sh(u, a, 0)
        for m in range(1, R + 1):
            torch.add(_sh(u, a, m), _sh(u, a, -m), out=self.tmp)
            self.tmp.sub_(c, alpha=2.0)
            out.add_(self.tmp, alpha=self.w[m - 1])
        return out

    def lap(self, u):
        if self.case["surface"]:
            _odd_image(u)
        self.L.zero_()
        c = _sh(u, 0, 0)
        for a in range(3):
            for m in range(1, R + 1):
                torch.add(_sh(u, a, m), _sh(u, a, -m), out=self.tmp)
                self.tmp.sub_(c, alpha=2.0)
                self.L.add_(self.tmp, alpha=self.w[m - 1])
        return self.L

    def step(self, up, u, pos, val):
        """u^{n+1} into up (holding u^{n-1}); val: what the numerator gains at the points pos."""
        lap = self.lap(u)
        lap.mul_(self.C)
        c, p = _sh(u, 0, 0), _sh(up, 0, 0)
        torch.sub(self.e, 1.0, out=self.tmp)
        p.mul_(self.tmp).add_(c, alpha=2.0).add_(lap)
        p.index_put_(pos, val, accumulate=True)
        torch.add(self.e, 1.0, out=self.tmp)
        p.div_(self.tmp)
        if self.case["surface"]:
            p[0] = 0.0


def _pos(ijk, dev):
    t = torch.from_numpy(ijk.astype(np.int64)).to(dev)
    return t[:, 2], t[:, 1], t[:, 0]


def _exact_forward(case, vel, src, rec, wav, keep=None):
    """(traces, final state); keep: gets g^n = L u^n + s^n of every step."""
    r = _Ref(case, vel)
    dev = r.dev
    ps, pr = _pos(src, dev), _pos(rec, dev)
    w = torch.from_numpy(wav).double().to(dev)
    a, b = _padded(r.shape, dev), _padded(r.shape, dev)
    cell = H ** 3
    traces = torch.empty((case["nt"], len(rec)), dtype=torch.float64, device=dev)
    for n in range(case["nt"]):
        if keep is not None:
            g = r.lap(b).clone()
            g.index_put_(ps, w[:, n] / cell, accumulate=True)
            if case["surface"]:
                g[0] = 0.0
            keep.append(g)
        r.step(a, b, ps, r.C[ps] * w[:, n] / cell)
        a, b = b, a
        traces[n] = _sh(b, 0, 0)[pr]
    return traces, _sh(b, 0, 0).contiguous()


def _exact_backward(case, vel, src, rec, resid, g=None):
    """(adjoint sources [nsrc][nt], velocity gradient or None) of the residual [nt][nrec]."""
    r = _Ref(case, vel)
    dev = r.dev
    ps, pr = _pos(src, dev), _pos(rec, dev)
    res = resid.double()
    a, b = _padded(r.shape, dev), _padded(r.shape, dev)
    adj = torch.empty((len(src), case["nt"]), dtype=torch.float64, device=dev)
    acc = torch.zeros(r.shape, dtype=torch.float64, device=dev) if g is not None else None
    for n in range(case["nt"] - 1, -1, -1):
        r.step(a, b, pr, r.C[pr] * res[n])
        a, b = b, a
        psi = _sh(b, 0, 0)
        adj[:, n] = psi[ps] / H ** 3
        if g is not None:
            acc.addcmul_(psi, g[n])
    return adj, None if g is None else 2.0 * acc / r.vel


def _memory(r, a, f0, half):
    """CPML coefficients b, g of axis a at the grid points (half: the half points), shaped to broadcast."""
    n, nbl = r.shape[a], r.case["nbl"]
    s = r.depth(a, np.arange(n) + 0.5 * half) / nbl
    d = 3.0 * r.vmax * math.log(1.0 / REFL) / (2.0 * nbl * H) * s * s
    al = math.pi * f0 * (1.0 - s)
    b = np.where(s > 0, np.exp(-(d + al) * DT), 1.0)
    g = np.where(s > 0, d * (b - 1.0) / np.where(s > 0, d + al, 1.0), 0.0)
    shape = [1, 1, 1]
    shape[a] = n
    return (torch.from_numpy(np.ascontiguousarray(x)).to(r.dev).reshape(shape) for x in (b, g))


def _exact_cpml(case, vel, src, rec, wav):
    r = _Ref(case, vel)
    dev, cell = r.dev, H ** 3
    ps, pr = _pos(src, dev), _pos(rec, dev)
    w = torch.from_numpy(wav).double().to(dev)
    up, u = _padded(r.shape, dev), _padded(r.shape, dev)
    psi, zeta = [_padded(r.shape, dev) for _ in range(3)], [torch.zeros(r.shape, dtype=torch.float64, device=dev) for _ in range(3)]
    bg = [tuple(_memory(r, a, F0, 0)) for a in range(3)]
    traces = torch.empty((case["nt"], len(rec)), dtype=torch.float64, device=dev)

    def d1(f, a):
        out = torch.zeros(r.shape, dtype=torch.float64, device=dev)
        for m in range(1, R + 1):
            out.add_(_sh(f, a, m) - _sh(f, a, -m), alpha=FIRST[m - 1] / H)
        return out

    for n in range(case["nt"]):
        if case["surface"]:
            _odd_image(u)
        total = torch.zeros(r.shape, dtype=torch.float64, device=dev)
        for a in range(3):
            b, g = bg[a]
            on = g != 0.0
            q = _sh(psi[a], 0, 0)
            q.mul_(b).add_(g * d1(u, a))
            # the correction acts inside the layers only
            extra = d1(psi[a], a) * on
            d2 = r.axis_term(u, a, r.L)
            zeta[a].mul_(b).add_(g * (d2 + extra))
            total += d2
            total += extra
            total += zeta[a]
        p = _sh(up, 0, 0)
        p.neg_().add_(_sh(u, 0, 0), alpha=2.0).addcmul_(r.C, total)
        p.index_put_(ps, r.C[ps] * w[:, n] / cell, accumulate=True)
        if case["surface"]:
            p[0] = 0.0
        up, u = u, up
        traces[n] = _sh(u, 0, 0)[pr]
    return traces, _sh(u, 0, 0).contiguous()


def _exact_vd(case, vel, rho, src, rec, wav):
    r = _Ref(case, vel)
    dev, cell = r.dev, H ** 3
    ps, pr = _pos(src, dev), _pos(rec, dev)
    w = torch.from_numpy(wav).double().to(dev)
    rho = rho.double()
    K = rho * r.vel * r.vel
    p, v = _padded(r.shape, dev), [_padded(r.shape, dev) for _ in range(3)]
    half_b, e_half, nbl = [], [], case["nbl"]
    eta_max = 3.0 * r.vmax * math.log(1.0 / REFL) / (2.0 * nbl * H)

    def eta(a, half):
        x = r.depth(a, np.arange(r.shape[a]) + 0.5 * half) / nbl
        shape = [1, 1, 1]
        shape[a] = r.shape[a]
        return torch.from_numpy(DT * eta_max * x * x).to(dev).reshape(shape)

    for a in range(3):
        b = 1.0 / rho
        nxt = torch.cat([b.narrow(a, 1, b.shape[a] - 1), b.narrow(a, b.shape[a] - 1, 1)], a)
        half_b.append(0.5 * (b + nxt))
        e_half.append(sum(eta(c, 1 if c == a else 0) for c in range(3)))
    e0 = sum(eta(c, 0) for c in range(3))
    if case["cpml"]:
        hb, gb = [tuple(_memory(r, a, F0, 1)) for a in range(3)], [tuple(_memory(r, a, F0, 0)) for a in range(3)]
        psi = [torch.zeros(r.shape, dtype=torch.float64, device=dev) for _ in range(3)]
        phi = [torch.zeros(r.shape, dtype=torch.float64, device=dev) for _ in range(3)]
        e0 = torch.zeros((1, 1, 1), dtype=torch.float64, device=dev)
    e_src = e0.expand(r.shape)[ps]
    traces = torch.empty((case["nt"], len(rec)), dtype=torch.float64, device=dev)

    def diff(f, a, forward):
        out = torch.zeros(r.shape, dtype=torch.float64, device=dev)
        for m in range(1, R + 1):
            hi, lo = (m, 1 - m) if forward else (m - 1, -m)
            out.add_(_sh(f, a, hi) - _sh(f, a, lo), alpha=STAGGERED[m - 1] / H)
        return out

    for n in range(case["nt"]):
        if case["surface"]:
            _odd_image(p)
        for a in range(3):
            dp, x = diff(p, a, True), _sh(v[a], 0, 0)
            if case["cpml"]:
                psi[a].mul_(hb[a][0]).add_(hb[a][1] * dp)
                x.add_(DT * half_b[a] * (dp + psi[a]))
            else:
                x.mul_(1.0 - 0.5 * e_half[a]).add_(DT * half_b[a] * dp).div_(1.0 + 0.5 * e_half[a])
        if case["surface"]:
            for m in range(1, R + 1):
                v[0][R - m] = v[0][R + m - 1]
        div = torch.zeros(r.shape, dtype=torch.float64, device=dev)
        for a in range(3):
            dv = diff(v[a], a, False)
            div += dv
            if case["cpml"]:
                phi[a].mul_(gb[a][0]).add_(gb[a][1] * dv)
                div += phi[a]
        x = _sh(p, 0, 0)
        x.mul_(1.0 - 0.5 * e0).add_(DT * K * div).div_(1.0 + 0.5 * e0)
        x.index_put_(ps, DT * K[ps] * w[:, n] / (cell * (1.0 + 0.5 * e_src)), accumulate=True)
        if case["surface"]:
            x[0] = 0.0
        traces[n] = x[pr]
    # the library's order of the components: p, vx, vy, vz
    return traces, torch.stack([_sh(f, 0, 0) for f in (p, v[2], v[1], v[0])])


def exact(case, seed):
    """What run() returns, in 64 bits."""
    if case["kind"] == "batch":
        out = []
        for s, c in enumerate(_shots(case)):
            vel, src, rec, wav = _inputs(c, seed + 100 * s)
            out.append(_exact_forward(c, vel, src, rec, wav)[0])
        return out
    vel, src, rec, wav = _inputs(case, seed)
    kind = case["kind"]
    if kind == "vd":
        return _exact_vd(case, vel, _density(vel, seed), src, rec, wav)
    if kind == "forward":
        return (_exact_cpml if case["cpml"] else _exact_forward)(case, vel, src, rec, wav)
    resid = _residual(case, len(rec), seed)
    if kind == "adjoint":
        return _exact_backward(case, vel, src, rec, resid)[0]
    keep = []
    traces, _ = _exact_forward(case, vel, src, rec, wav, keep)
    if kind == "gradient":
        return _exact_backward(case, vel, src, rec, resid, keep)[1]
    adj, gv = _exact_backward(case, vel, src, rec, traces - resid.double(), keep)
    return traces, gv, adj
