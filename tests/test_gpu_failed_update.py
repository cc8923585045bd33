"""mbd_update_positions with every growing allocation failing in turn (a denser geometry
whose pair list outgrows its buffers): MBD_ERR_OOM, then every call that reads
the geometry is refused instead of reading lists that are gone, and an update that
succeeds gives bit for bit the results of before."""
import ctypes

import numpy as np
import pytest
import torch

from workloads.systems import water_system

pytestmark = pytest.mark.gpu

INVALID_ARG, OOM = 1, 2


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_failed_update(mbd, precision):
    from paper_2307_02278_gb300._abi import lib as load
    lib = load()
    s = water_system(300, 17, mesh=(48, 48, 48))
    n = s.n_atoms
    centre = s.cell.sum(axis=0) / 2
    dense = centre + 0.8 * (np.mod(s.pos, np.diag(s.cell)) - centre)
    x = torch.randn(4, 3 * n, dtype=torch.float64, device="cuda")
    d = x.reshape(4, n, 3)
    failures = 0
    for k in range(50):
        g = mbd.MBDSystem.from_workload(s, precision=precision)
        y, (e, f) = g.apply_C(x), g.energy_forces(4, 6, 3)
        lib.mbd_debug_fail_allocation(k)
        rc = lib.mbd_update_positions(g._handle, dense.ctypes.data_as(ctypes.POINTER(ctypes.c_double)))
        lib.mbd_debug_fail_allocation(-1)
        if rc == 0:
            g.close()
            break
        assert rc == OOM
        failures += 1
        for call in (lambda: g.apply_C(x), lambda: g.field(d), lambda: g.spread(d, s.mesh), lambda: g.autotune(4),
                     lambda: g.lanczos_energy(4, 6, 3), lambda: g.energy_forces(4, 6, 3), lambda: g.scs_screen(8)):
            with pytest.raises(mbd.MBDError) as err:
                call()
            assert err.value.code == INVALID_ARG
        g.update_positions(s.pos)
        e2, f2 = g.energy_forces(4, 6, 3)
        assert torch.equal(g.apply_C(x), y) and e2 == e and torch.equal(f2, f)
        g.close()
    assert failures >= 6           # neighbours, shifts, both tensors, cluster entries and records
