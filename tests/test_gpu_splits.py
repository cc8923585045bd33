"""The kernels' splits over lanes, warps and pencils, at the probe counts and spline
orders where they change: probes that fill a lane's 16 bytes, a warp, a
64-probe chunk or two, and one more; every spline order; the real space in the
field kernel and on clusters; a skew cell with a mesh of three lengths.  Against
the oracle at the tolerances of the parity tests (FP64 1e-11 for products, 1e-8
for quadratures and forces; FP32 operator 2e-6, forces 1e-4).  The neighbour
list is compared by its pair count with pairs a few 1e-9 bohr on either side of
the cutoff, which its FP32 prefilter must all pass on."""
import numpy as np
import pytest
import torch

from _parity import close
from oracle.ewald import pair_list
from oracle.forces import estimator_forces
from oracle.lanczos import slq
from oracle.operator import Operator
from workloads.systems import System, random_system

pytestmark = pytest.mark.gpu

PRODUCT_TOL = {"fp64": 1e-11, "mixed": 2e-6}
Q_TOL = {"fp64": 1e-8, "mixed": 2e-6}
FORCE_TOL = {"fp64": 1e-8, "mixed": 1e-4}


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


def _skew(order, n=70):
    s = random_system(n, 18.0, 515, mesh=(20, 27, 24), r_cut=7.9, damp_cut=7.9, spline_order=order)
    cell = s.cell @ np.array([[1.0, 0.0, 0.0], [0.1, 1.0, 0.0], [-0.05, 0.12, 1.0]])
    return s.with_(cell=cell, pos=(s.pos / 18.0) @ cell)


@pytest.fixture(scope="module")
def operators():
    return {p: (s, Operator(s, "spme")) for p in (4, 6, 8, 10) for s in [_skew(p)]}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("method", ["pairs", "clusters"])
@pytest.mark.parametrize("order", [4, 6, 8, 10])
def test_products(mbd, operators, order, method, precision):
    s, op = operators[order]
    g = mbd.MBDSystem.from_workload(s, precision=precision)
    g.set_real_space_method(method)
    x = np.random.default_rng(order).normal(size=(130, 3 * s.n_atoms))
    ref = op(x)
    for nvec in (1, 2, 3, 5, 16, 31, 33, 63, 64, 65, 128, 130):
        y = g.apply_C(torch.tensor(x[:nvec], device="cuda")).cpu().numpy()
        close(y, ref[:nvec], PRODUCT_TOL[precision])
    g.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("probes", [1, 2, 3, 7, 16, 31, 32, 33, 65])
def test_quadratures(mbd, operators, probes, precision):
    """The prologue's rows per warp, the reductions over blocks and the register
    slots of the quadrature (33 steps: two)."""
    s, op = operators[6]
    g = mbd.MBDSystem.from_workload(s, precision=precision)
    for steps in (5, 33):
        _, det = g.lanczos_energy(probes, steps, 41, details=True)
        q_ref, _, _, _ = slq(op, 3 * s.n_atoms, probes, steps, 41)
        np.testing.assert_allclose(det["q"], q_ref, rtol=Q_TOL[precision])
    g.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("order", [4, 6, 8, 10])
def test_forces(mbd, operators, order, precision):
    s, op = operators[order]
    g = mbd.MBDSystem.from_workload(s, precision=precision)
    for probes in (1, 3, 17, 65):
        _, f = g.energy_forces(probes, 6, 43)
        f_ref, _, _ = estimator_forces(op, probes, 6, 43)
        assert np.abs(f.cpu().numpy() - f_ref).max() <= FORCE_TOL[precision] * np.abs(f_ref).max()
    g.close()


def test_neighbours_at_the_cutoff(mbd):
    """A lattice whose fifth shell lies at the cutoff, shifted by a few 1e-9 bohr
    per atom, far from the origin of a long cell."""
    rng = np.random.default_rng(3)
    edge, a = np.array([120.0, 20.0, 20.0]), 4.0
    grid = np.stack(np.meshgrid(*[np.arange(int(e / a)) for e in edge], indexing="ij"), -1).reshape(-1, 3)
    pos = (grid + 0.5) * a + rng.uniform(-4e-9, 4e-9, (len(grid), 3))
    n = len(pos)
    s = System("lattice", np.diag(edge), pos, np.full(n, 5.0), np.full(n, 0.5), np.full(n, 3.2), r_cut=2.0 * a,
               damp_cut=2.0 * a, mesh=(120, 20, 20))
    g = mbd.MBDSystem.from_workload(s, precision="fp64")
    i, _, r = pair_list(s.cell, s.pos, s.r_cut)
    at_cutoff = np.abs(np.linalg.norm(r, axis=1) - s.r_cut) < 1e-7
    assert 0 < at_cutoff.sum() < 6 * n
    assert g.info()["n_pairs"] == len(i)
    g.close()
