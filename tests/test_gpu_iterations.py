"""Blocks that take several atoms at once and several iterations, and the spreading's
longer segments: branches that systems of a hundred atoms and a few hundred tiles
do not reach.

- 2502 atoms (a multiple of no atoms per block but 1, 2, 3, 6 and 9): blocks of the field
  kernels take 3 (33 and 36 FP32 probes), 4, 8 and more atoms at once, and the streamed
  kernel crosses atoms and its weight buffers.  Products against the oracle at the
  tolerances of the parity tests (FP64 1e-11, FP32 operator 2e-6); the atoms per block,
  forced from one to 64, do not change a bit of them, and the coefficients of a
  short run only by the order of their sums (FP64 1e-12, FP32 operator 1e-6).
- 48 x 48 pencils x 64 probes (32 in double): more than eight tiles per SM, so four and
  six segments per pencil; products of the same vectors eight at a time (up to eight
  segments, which the other tests compare with the oracle) within 1e-12 and 2e-6."""
import numpy as np
import pytest
import torch

from _parity import close
from oracle.operator import Operator
from workloads.systems import random_system, water_system

pytestmark = pytest.mark.gpu

PRODUCT_TOL = {"fp64": 1e-11, "mixed": 2e-6}


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.fixture(scope="module", params=[4, 6, 8, 10])
def box(request):
    order = request.param
    s = water_system(834, 23, r_cut=9.0, damp_cut=9.0, ewald_beta=0.35, mesh=(54, 60, 50), spline_order=order)
    x = np.random.default_rng(order).normal(size=(132, 3 * s.n_atoms))
    return s, x, Operator(s, "spme")(x)


@pytest.mark.parametrize("method", ["pairs", "clusters"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_several_atoms_per_block(mbd, box, precision, method):
    s, x, ref = box
    g = mbd.MBDSystem.from_workload(s, precision=precision)
    g.set_real_space_method(method)
    for nvec in (1, 5, 12, 33, 36, 64, 100, 132):
        xd = torch.tensor(x[:nvec], device="cuda")
        g.set_launch_choices(None)
        y = g.apply_C(xd)
        close(y.cpu().numpy(), ref[:nvec], PRODUCT_TOL[precision])
        for apb in (1, 7, 64):
            g.set_launch_choices({"ld": nvec + nvec % 2, "field_atoms_per_block": apb})
            assert torch.equal(g.apply_C(xd), y), (nvec, apb)
    tol = 1e-12 if precision == "fp64" else 1e-6
    for probes in (3, 36, 64):
        g.set_launch_choices(None)
        _, d0 = g.lanczos_energy(probes, 4, 9, details=True)
        for apb in (1, 7, 64):
            g.set_launch_choices({"ld": probes + probes % 2, "field_atoms_per_block": apb})
            _, d1 = g.lanczos_energy(probes, 4, 9, details=True)
            np.testing.assert_allclose(d1["a"], d0["a"], rtol=tol)
    g.close()


def _smooth(n):
    for f in (2, 3, 5):
        while n % f == 0:
            n //= f
    return n == 1


@pytest.mark.parametrize("order", [4, 6, 8, 10])
@pytest.mark.parametrize("precision,nvec,tol", [("fp64", 32, 1e-12), ("mixed", 64, 2e-6)])
def test_many_tiles(mbd, precision, nvec, tol, order):
    bad = []
    for k in [k for k in range(max(16, 2 * order), 201) if _smooth(k)]:
        s = random_system(40, 18.0, 99, mesh=(48, 48, k), r_cut=7.9, damp_cut=7.9, spline_order=order)
        g = mbd.MBDSystem.from_workload(s, precision=precision)
        x = torch.tensor(np.random.default_rng(k).normal(size=(nvec, 3 * s.n_atoms)), device="cuda")
        y = g.apply_C(x)
        few = torch.cat([g.apply_C(x[v:v + 8].contiguous()) for v in range(0, nvec, 8)])
        err = float((y - few).norm() / few.norm())
        if not err < tol:
            bad.append((k, err))
        g.close()
    assert not bad, bad
