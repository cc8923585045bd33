"""A dipole that is not finite reaches the real-space field of its neighbours and of
nobody else, on the clusters (whose records serve two atoms, one of which may not
be a neighbour) as in the pair loop.  The atoms concerned come from the pair list;
the others' fields are those with a dipole of zero in its place, bit for bit."""
import numpy as np
import pytest
import torch

from oracle.ewald import pair_list
from workloads.systems import water_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e200])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("method", ["clusters", "pairs"])
def test_neighbours_only(mbd, method, precision, value):
    if value == 1e200 and precision == "fp64":
        pytest.skip("finite in double")
    s = water_system(200, 5, r_cut=6.0, damp_cut=6.0, mesh=(32, 32, 32))
    at = 123
    i, j, _ = pair_list(s.cell, s.pos, s.r_cut)
    reached = np.zeros(s.n_atoms, bool)
    reached[i[j == at]] = True
    assert 5 < reached.sum() < 100
    for nvec in (1, 5, 40):
        d = np.random.default_rng(2).normal(size=(nvec, s.n_atoms, 3))
        d[:, at] = 0.0
        g = mbd.MBDSystem.from_workload(s, precision=precision)
        g.set_real_space_method(method)
        plain = g.field(torch.tensor(d, device="cuda"), 1).cpu().numpy()
        d[:, at] = value
        e = g.field(torch.tensor(d, device="cuda"), 1).cpu().numpy()
        finite = np.isfinite(e).all(axis=2)
        assert np.array_equal(finite, np.broadcast_to(~reached, finite.shape))
        assert np.array_equal(e[:, ~reached], plain[:, ~reached])
        g.close()
