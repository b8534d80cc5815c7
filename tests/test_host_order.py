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


H2D = 1   # cudaMemcpyHostToDevice


def _uploads_done(log):
    """Every upload or fill of a set-up call was waited for before the call returned;
    the streams they ran on (0: the legacy stream, which orders nothing for
    non-blocking streams)."""
    last = {}
    for i, e in enumerate(log):
        if e["op"] == "memset" or e["op"] == "memcpy" and e["kind"] == H2D:
            last[e["stream"]] = i
    for stream, i in last.items():
        assert any(e["op"] == "sync" and e["stream"] == stream for e in log[i:]), stream
    return set(last)


def _stays_on(log, stream):
    """Nothing of a run is allocated, uploaded or put on another caller's stream."""
    for e in log:
        assert e["op"] != "malloc" and not (e["op"] == "memcpy" and e["kind"] == H2D), e
        assert e.get("stream", stream) != 0, e


def test_create_returns_with_its_tables_in_place(rt):
    rt.log()
    p = _problem(shape=(40, 100, 130))
    rt.propagator(p, model=False)
    assert _uploads_done(rt.log())


@pytest.mark.parametrize("change", [("variant", v) for v in (9, 10, 11, 0, -1)]
                         + [("option", (M.OPT_PERSISTENT, 1)), ("option", (M.OPT_CLAIM, 4))])
def test_another_tile_shape_is_set_up_by_the_call_that_selects_it(rt, change):
    """Tables of another tile shape are complete when the selecting call returns;
    the runs that follow, on any stream, allocate and upload nothing."""
    p = _problem(shape=(40, 100, 130))
    prop = rt.propagator(p)
    assert prop.plan()["variant"] == 9   # 48 x 20 tiles: the options below need 64 x 16
    wav, traces, resid, adj, grad = (rt.malloc(n) for n in (p.wavelet.size, p.nt * 9, p.nt * 9, p.nt * 2, p.vel.size))
    s = rt.stream()

    def runs():
        prop.forward(wav, traces, stream=s)
        prop.adjoint(resid, adj, stream=s)
        prop.gradient(wav, resid, grad, 4, M.CKPT_BF16, stream=s)

    runs()
    rt.log()
    kind, value = change
    prop.set_variant(value) if kind == "variant" else prop.set_option(*value)
    built = _uploads_done(rt.log())
    assert 0 not in built and len(built) == (0 if change in (("variant", 9), ("variant", -1)) else 1)
    runs()
    _stays_on(rt.log(), s)


@pytest.mark.parametrize("mode,variant", [(M.BATCH_FUSED, None), (M.BATCH_PERSISTENT, None), (M.BATCH_STREAMS, 5)])
def test_batch_sets_up_its_tiles(rt, mode, variant):
    p = _problem(shape=(40, 100, 130))
    props = [rt.propagator(p) for _ in range(2)]
    b = rt.batch(props)
    bufs = [[rt.malloc(n) for _ in props] for n in (p.wavelet.size, p.nt * 9)]
    rt.log()
    b.set_mode(mode)
    if variant is not None:
        b.set_variant(variant)
    assert _uploads_done(rt.log()) - {0}
    s = rt.stream()
    b.forward(*bufs, stream=s)
    log = rt.log()
    assert not [e for e in log if e["op"] == "malloc"]
    assert all(e["stream"] != 0 for e in log if "stream" in e)   # the shots' arguments go up on the caller's


@pytest.mark.parametrize("scheme,dtype,ckpt", [(M.SCHEME_SEGMENTS, M.CKPT_FP32, 4), (M.SCHEME_SEGMENTS, M.CKPT_FP32, 16),
                                               (M.SCHEME_SEGMENTS, M.CKPT_BF16, 4), (M.SCHEME_REVOLVE, M.CKPT_FP32, 3)])
def test_first_gradient_fills_its_work_volumes_on_the_callers_stream(rt, scheme, dtype, ckpt):
    p = _problem()
    prop = rt.propagator(p)
    prop.set_option(M.OPT_CKPT_SCHEME, scheme)
    wav, resid, grad = (rt.malloc(n) for n in (p.wavelet.size, p.nt * 9, p.vel.size))
    s = rt.stream()
    rt.log()
    prop.gradient(wav, resid, grad, ckpt, dtype, stream=s)
    assert all(e["stream"] != 0 for e in rt.log() if "stream" in e)


@pytest.mark.parametrize("make", ["batch", "vd", "vd_cpml"])
def test_batches_and_staggered_handles_return_with_their_tables_in_place(rt, make):
    if make == "batch":
        props = [rt.propagator(_problem(), model=False)]
        rt.log()
        rt.batch(props)
    else:
        p = W.tiny_problem_vd(shape=(12, 30, 40), nt=16, nbl=4, nsrc=3, nrec=9, seed=3)
        p.cpml, p.cpml_f0 = make == "vd_cpml", 15.0 if make == "vd_cpml" else 0.0
        rt.log()
        rt.open.append(M.StaggeredPropagator.from_problem(p))
    assert _uploads_done(rt.log())


@pytest.mark.parametrize("mode", [M.BATCH_STREAMS, M.BATCH_FUSED])
@pytest.mark.parametrize("fast", ["StagedILi48", "StagedILi40", "StagedILi32", "StagedILi64", "5ShapeILi16ELi2ELi1"])
def test_a_tuned_batch_variant_can_be_set_again(rt, fast, mode):
    """Whatever kernel turns out fastest, the number that tuning returns is taken by
    set_variant and selects what tuning left selected."""
    props = [rt.propagator(_problem(shape=shape)) for shape in ((64, 64, 64), (40, 100, 130))]

    def variants():
        return [pr.plan()["variant"] for pr in props]

    own = variants()
    assert own == [2, 9]
    b = rt.batch(props)
    b.set_mode(mode)
    rt.lib.fake_fast_kernel(fast.encode())
    v = b.autotune(steps=3)
    tuned = variants()
    b.set_variant(v)
    if mode == M.BATCH_STREAMS:   # tuning the fused kernels leaves the shots' own loops alone
        assert variants() == tuned and (v == 2 or fast != "StagedILi48")
    b.set_variant(5)
    assert variants() == [5, 5]
    b.set_variant(2)   # the default form: each shot in its own tile shape
    assert variants() == own


@pytest.mark.parametrize("dtype", [M.CKPT_FP32, M.CKPT_BF16])
@pytest.mark.parametrize("nth", range(1, 9))
def test_work_volume_maps_after_a_failed_change_of_tiles(rt, nth, dtype):
    """The work volumes' tensor maps are encoded anew for another tile shape; if that
    fails half way, a later run in the old shape must not use what was encoded."""
    prop = rt.propagator(_problem(shape=(40, 100, 130)))
    wav, resid, grad = (rt.malloc(n) for n in (2 * 16, 16 * 9, 40 * 100 * 130))

    def gradient():
        prop.gradient(wav, resid, grad, 8, dtype)

    prop.set_variant(9)
    gradient()
    prop.set_variant(10)
    prop.set_variant(9)   # both shapes of the handle's own volumes are set up
    prop.set_variant(10)
    rt.lib.fake_fail_encode(0, 0, nth)
    with pytest.raises(M.MmodError):
        gradient()
    rt.lib.fake_fail_encode(0, 0, 0)
    prop.set_variant(9)
    rt.log()
    gradient()
    boxes = {}
    for e in rt.log():
        if e["op"] == "encode":
            boxes[e["map"]] = tuple(e["box"])
    # every map overwritten for the 40 x 24 tiles is one of the 48 x 20 tiles again
    assert len(boxes) >= nth - 1 and set(boxes.values()) <= {(56, 28), (48, 20)}
    assert {(56, 28), (48, 20)} <= set(boxes.values())


def _step_kernels(rt, prop, p):
    rt.log()
    prop.forward(rt.malloc(p.wavelet.size), rt.malloc(p.nt * 9))
    names = {e["name"] for e in rt.log() if e["op"] == "launch"}
    return {n for n in names if "step_tma_kernel" in n or "step_simple_kernel" in n}


@pytest.mark.parametrize("box", [(56, 28), (48, 20)])
def test_create_falls_back_to_the_default_tiles(rt, box):
    """Tile shapes whose maps cannot be encoded give way to 64 x 16, not to the plain kernel."""
    p = _problem(shape=(40, 100, 130))
    rt.lib.fake_fail_encode(*box, 1)
    prop = rt.propagator(p)
    assert prop.plan()["variant"] == 2
    kernels = _step_kernels(rt, prop, p)
    assert kernels and all("StagedILi64" in k for k in kernels)
    with pytest.raises(M.MmodError) as ei:   # the shape itself stays refused, and selecting it changes nothing
        prop.set_variant(9)
    assert ei.value.status == -7 and prop.plan()["variant"] == 2


def test_create_falls_back_to_the_plain_kernel(rt):
    p = _problem(shape=(40, 100, 130))
    rt.lib.fake_fail_encode(0, 0, 1)
    prop = rt.propagator(p)
    kernels = _step_kernels(rt, prop, p)
    assert kernels and all("step_simple_kernel" in k for k in kernels)


@pytest.mark.parametrize("entries", [40 * 3 * 5 + 1, 40 * 3 * 7 + 1])   # bucket starts of 48 x 20 and of 64 x 16 tiles
def test_create_reports_memory_that_is_missing_for_tables(rt, entries):
    rt.lib.fake_fail_malloc(4 * entries)
    with pytest.raises(M.MmodError) as ei:
        rt.propagator(_problem(shape=(40, 100, 130)))
    assert M.STATUS[ei.value.status].endswith("OOM")


@pytest.mark.parametrize("first,second", [({M.OPT_CPML_TILES: 1}, {M.OPT_CPML_TILES: 0}),
                                          ({M.OPT_ZLEN: 1 << 19}, {M.OPT_ZLEN: 0, M.OPT_CLAIM: 1}),
                                          ({M.OPT_CLAIM: 1 << 20}, {M.OPT_CLAIM: 0, M.OPT_CPML_PLANES: 1}),
                                          ({M.OPT_PDL: 0}, {M.OPT_PDL: 1}), ({M.OPT_ZLEN: 4}, {M.OPT_ZLEN: 5})])
def test_an_option_changed_between_runs_takes_effect(rt, first, second):
    """Every option that the captured loop depends on makes the next run capture anew."""
    p = _problem()
    p.cpml, p.cpml_f0, p.nbl = True, 15.0, 4
    prop = rt.propagator(p)
    prop.set_variant(2)   # the same kernel throughout
    wav, tr = rt.malloc(p.wavelet.size), rt.malloc(p.nt * 9)
    for options, captures in ((first, 1), (first, 0), (second, 1), (second, 0)):
        for o, v in options.items():
            prop.set_option(o, v)
        rt.log()
        prop.forward(wav, tr)
        assert len([e for e in rt.log() if e["op"] == "begin_capture"]) == captures


def test_tuning_skips_tiles_that_cannot_be_set_up(rt):
    """A handle that fell back to the default tiles can still be tuned, and runs afterwards."""
    p = _problem(shape=(40, 100, 130))
    rt.lib.fake_fail_encode(48, 20, 1)
    prop = rt.propagator(p)
    rt.lib.fake_fast_kernel(b"StagedILi40")
    assert prop.autotune(steps=3) == 10
    kernels = _step_kernels(rt, prop, p)
    assert kernels and all("StagedILi40" in k for k in kernels)
