"""Mesh lengths without a compiled pass (below 16, or not among the compiled ones up
to 256, or above): spreading with pencils cut into segments (few tiles) and whole
(many), transforms from one column per row on, and C x, against the
oracle: 1e-12 for FP64 transforms, 1e-11 for FP64 products, 1e-5 and 2e-6 with
the FP32 operator.  Spreading at the tolerances of the products."""
import numpy as np
import pytest
import torch

from _parity import atom_max, close, rel
from oracle import spme as ospme
from oracle.operator import Operator
from workloads.systems import random_system

pytestmark = pytest.mark.gpu

PRODUCT_TOL = {"fp64": 1e-11, "mixed": 2e-6}
FFT_TOL = {"fp64": 1e-12, "mixed": 1e-5}
# (mesh, order): the shortest and longest pencils for each order, odd lengths and uneven segments
MESHES = [((8, 10, 8), 4), ((9, 8, 15), 4), ((12, 12, 12), 6), ((15, 12, 15), 6), ((16, 20, 18), 8), ((20, 24, 20), 10),
          ((12, 15, 270), 6), ((12, 288, 12), 6), ((300, 12, 12), 4), ((20, 20, 324), 10)]


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


def _system(mesh, order):
    return random_system(90, 20.0, 99, mesh=mesh, r_cut=7.9, damp_cut=7.9, spline_order=order)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("mesh,order", MESHES)
def test_generic_lengths(mbd, mesh, order, precision):
    """1 to 5 probes: rows of one or two columns, several pencils per tile; 40: partial
    tiles; 300 on the small meshes: whole pencils per warp."""
    s = _system(mesh, order)
    op = Operator(s, "spme")
    g = mbd.MBDSystem.from_workload(s, precision=precision)
    rng = np.random.default_rng(order)
    for nvec in (1, 2, 3, 5, 40) + ((300,) if max(mesh) < 16 else ()):
        x = rng.normal(size=(nvec, 3 * s.n_atoms))
        close(g.apply_C(torch.tensor(x, device="cuda")).cpu().numpy(), op(x), PRODUCT_TOL[precision])
        d = x.reshape(nvec, s.n_atoms, 3)
        close(g.spread(torch.tensor(d, device="cuda"), mesh).cpu().numpy(), ospme.spread(s, d), PRODUCT_TOL[precision], width=1)
        q = rng.normal(size=(nvec,) + mesh)
        phi, ref = g.convolve(torch.tensor(q, device="cuda")).cpu().numpy(), ospme.convolve(s, q)
        assert rel(phi, ref) < FFT_TOL[precision] and atom_max(phi, ref, width=1) < 10.0 * FFT_TOL[precision]
    g.close()
