"""Screening of a matrix that is not positive definite (the polarisation catastrophe,
from enlarged polarisabilities): MBD_ERR_NOT_POSITIVE_DEFINITE, outputs untouched,
and the call ends once the curvature test has failed, however many iterations it
was allowed (at most four more are queued).  One block per atom (450 atoms) and
one warp per atom (6000), both precisions."""
import ctypes
import time

import numpy as np
import pytest
import torch

from workloads.systems import water_system

pytestmark = pytest.mark.gpu

NOT_POSITIVE_DEFINITE = 4


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


def _screen(lib, g, n, max_iter):
    out = [np.full(n, 7.0) for _ in range(3)]
    p = [x.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for x in out]
    t0 = time.perf_counter()
    st = lib.mbd_scs_screen(g._handle, 15, 1e-10, max_iter, p[0], p[1], p[2], None, None, None, None)
    return st, time.perf_counter() - t0, out


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("molecules", [150, 2000])
def test_not_positive_definite(mbd, molecules, precision):
    from paper_2307_02278_gb300._abi import lib
    s = water_system(molecules, 77, r_cut=9.0, damp_cut=9.0, ewald_beta=0.35)
    big = s.with_(alpha=40.0 * s.alpha)
    with mbd.MBDSystem.from_workload(big, precision=precision) as g:
        few = [_screen(lib(), g, s.n_atoms, 200) for _ in range(2)][1]
        many = _screen(lib(), g, s.n_atoms, 100000)
    for st, _, out in (few, many):
        assert st == NOT_POSITIVE_DEFINITE
        assert all(np.all(x == 7.0) for x in out)
    # no more iterations than 200 would have run, let alone 100,000
    assert many[1] < 10.0 * few[1] + 0.1, (few[1], many[1])
