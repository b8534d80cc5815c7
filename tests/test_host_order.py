"""What the host enqueues and in which order, checked on a CUDA runtime without a
device (_host_runtime.py)."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _host_runtime import host_runtime


@pytest.fixture
def rt():
    with host_runtime() as r:
        yield r


def _problem(shape=(12, 30, 40), nt=16, nsrc=2, nrec=9):
    return W.tiny_problem(shape=shape, nt=nt, nbl=4, nsrc=nsrc, nrec=nrec, seed=3)


def _captured_records(log):
    """Trace-row events recorded inside the loop's capture (the first and the
    last record bracket the loop)."""
    return [e["event"] for e in log if e["op"] == "record" and e["capture"]][1:-1]


def test_host_traces_never_replay_a_loop_without_row_events(rt):
    """Device traces at an address that the staging buffer of host traces gets
    later: the download waits for row events, so the loop that records them
    must be captured although every pointer is the same."""
    p = _problem()
    prop = rt.propagator(p)
    wav = rt.malloc(p.wavelet.size)
    n = p.nt * len(p.rec_ijk)
    dev = rt.malloc(n)
    rt.log()
    prop.forward(wav, dev)
    assert not _captured_records(rt.log())
    rt.free(dev)
    prop.forward(wav, np.empty((p.nt, len(p.rec_ijk)), np.float32))
    log = rt.log()
    staging = [e["ptr"] for e in log if e["op"] == "malloc" and e["bytes"] == 4 * n]
    assert staging == [dev]   # the case in question
    rows = _captured_records(log)
    waits = [e["event"] for e in log if e["op"] == "wait"]
    assert rows and set(waits[:-1]) == set(rows)
    prop.forward(wav, np.empty((p.nt, len(p.rec_ijk)), np.float32))
    assert not [e for e in rt.log() if e["op"] == "begin_capture"]   # and is replayed from then on


def _launches(log):
    """The log with what a launch was given merged into the launch."""
    out = []
    for e in log:
        if e["op"] in ("step", "ckpt"):
            out[-1] = {**out[-1], **e}
        else:
            out.append(dict(e))
    return out


@pytest.mark.parametrize("scheme", [M.SCHEME_SEGMENTS, M.SCHEME_REVOLVE])
@pytest.mark.parametrize("dtype", [M.CKPT_FP32, M.CKPT_BF16, M.CKPT_FP16, M.CKPT_BFP16])
@pytest.mark.parametrize("ckpt", [1, 3, 5, 16])
def test_steps_read_early_only_what_is_settled(rt, ckpt, dtype, scheme):
    """A step with pdl 2 requests u^{n-1} and c before it waits for the operation
    in front of it: nothing there may write them (a restored checkpoint, a
    cleared volume, the step before)."""
    p = _problem()
    prop = rt.propagator(p)
    prop.set_option(M.OPT_CKPT_SCHEME, scheme)
    wav, resid, grad = (rt.malloc(n) for n in (p.wavelet.size, p.nt * len(p.rec_ijk), p.vel.size))
    rt.log()
    prop.gradient(wav, resid, grad, ckpt, dtype)
    written, steps, early = [], 0, 0
    for e in _launches(rt.log()):
        if e["op"] == "step":
            steps += 1
            if e["attrs"] and e["pdl"] == 2:
                early += 1
                for read in (e["uprev"], e["c"]):
                    assert not any(lo <= read < hi for lo, hi in written), (e, written)
            written = [(v, v + 1) for v in (e["uout"], e["gout"])]
        elif e["op"] == "ckpt":
            written = [(v, v + 1) for v in (e["u"] if e["restore"] else e["q"])]
        elif e["op"] in ("memset", "memcpy"):
            written = [(e["dst"], e["dst"] + e["bytes"])]
        elif e["op"] == "launch":
            written = []
    # three sweeps, or two where every state or term is kept; early reads are the rule in segments
    assert steps >= 2 * p.nt
    assert early >= (steps // 2 if scheme == M.SCHEME_SEGMENTS and ckpt < p.nt else 0)
