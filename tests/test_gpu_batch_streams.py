"""Streams of a batch: two for shots that fill the GPU, four for smaller ones, on
both sides of the line (mean points per shot 1.3e6) and with uneven shots:
every shot's bits as when it runs alone."""
import numpy as np
import pytest

import workloads as W
from _gpu_util import run_gpu
from test_gpu_batch import _run_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [[(109, 109, 109)] * 3, [(110, 110, 110)] * 3,
                                    [(30, 40, 50), (160, 200, 220), (24, 30, 33), (110, 128, 160), (20, 21, 22)],
                                    [(120, 120, 120)]])
def test_streams_bitwise(shapes):
    shots = [W.tiny_problem(shape=s, nt=15, nbl=5, nsrc=2, nrec=40, seed=i + 7) for i, s in enumerate(shapes)]
    tr_b, u_b, _ = _run_batch(shots)
    for i, p in enumerate(shots):
        tr_s, u_s, _ = run_gpu(p)
        assert np.array_equal(tr_b[i], tr_s) and np.array_equal(u_b[i], u_s), i
