"""What the host enqueues and in which order, checked on a CUDA runtime without a
device (_host_runtime.py)."""
import numpy as np
import pytest

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
