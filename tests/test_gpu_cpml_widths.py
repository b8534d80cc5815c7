"""Tiled CPML passes of every compiled layer width against the marching passes,
bit for bit: ragged along every line axis, x rows that are and are not 16-byte
aligned, two layers that just do not meet, with and without a free surface."""
import numpy as np
import pytest

import paper_2007_06048_gb300 as M
import workloads as W
from _gpu_util import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fs", [False, True])
@pytest.mark.parametrize("L", [8, 12, 16, 20, 24, 28, 32])
@pytest.mark.parametrize("extra", [(5, 7, 4), (13, 6, 5)])
def test_widths_bitwise(L, extra, fs):
    shape = tuple(2 * L + e for e in extra)
    p = W.tiny_problem(shape=shape, nt=30, nbl=L, nsrc=3, nrec=16, seed=L + extra[0])
    p.cpml, p.cpml_f0, p.free_surface = True, 25.0, fs
    p.src_ijk[0] = [2, shape[1] - 3, shape[0] - 2]
    p.rec_ijk[0] = [0, 0, shape[0] - 1]
    tr_m, u_m, _ = run_gpu(p, options={M.OPT_CPML_TILES: 0}, pdl=0)
    assert np.abs(u_m).max() > 0
    tr_t, u_t, _ = run_gpu(p, options={M.OPT_CPML_TILES: 1})
    assert np.array_equal(u_t, u_m) and np.array_equal(tr_t, tr_m)
