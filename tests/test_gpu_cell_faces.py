"""Atoms on the faces of non-orthogonal cells: crystals whose fractional coordinates
are exact fractions, zero among them.  In Cartesian coordinates and back, a
zero fraction is a rounding residue of either sign; the neighbour search must
put the atom into the search cell on the side where its position is.  The pair
count is compared with the brute-force count (no shell within 1e-6 of the
cutoff) and C x with the oracle's product, for a new system and for one whose
positions were updated, with three search cells or more in every direction."""
import numpy as np
import pytest
import torch

from _parity import close
from oracle.ewald import pair_list
from oracle.operator import Operator
from workloads.systems import System

pytestmark = pytest.mark.gpu

R_CUT = 8.13


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


def _supercell(name, prim, basis, reps):
    """`reps` primitive cells along each vector of prim, with the basis (fractions)."""
    cell = np.asarray(prim, float) * np.asarray(reps, float)[:, None]
    ijk = np.stack(np.meshgrid(*[np.arange(r) for r in reps], indexing="ij"), -1).reshape(-1, 3)
    frac = (ijk[:, None, :] + np.asarray(basis, float)[None]).reshape(-1, 3) / np.asarray(reps, float)
    pos = frac @ cell
    n = len(pos)
    return System(name, cell, pos, np.full(n, 5.0), np.full(n, 0.5), np.full(n, 3.2), r_cut=R_CUT, damp_cut=R_CUT,
                  mesh=(24, 24, 24))


def _systems():
    fcc = 4.0 * np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 1.0], [1.0, 1.0, 0.0]])
    a, c = 4.65, 12.68
    hexagonal = np.array([[a, 0.0, 0.0], [-a / 2, a * np.sqrt(0.75), 0.0], [0.0, 0.0, c]])
    graphite = [[0, 0, 0], [1 / 3, 2 / 3, 0], [0, 0, 0.5], [2 / 3, 1 / 3, 0.5]]
    monoclinic = np.array([[5.6, 0.0, 0.0], [0.0, 5.3, 0.0], [-1.7, 0.0, 5.5]])
    triclinic = np.array([[5.5, 0.3, -0.4], [0.9, 5.4, 0.2], [-1.3, 0.7, 5.7]])
    one = [[0, 0, 0]]
    return {"fcc": _supercell("fcc", fcc, one, (6, 6, 6)),
            "diamond": _supercell("diamond", fcc, [[0, 0, 0], [0.25, 0.25, 0.25]], (6, 6, 6)),
            "graphite": _supercell("graphite", hexagonal, graphite, (7, 7, 2)),
            "monoclinic": _supercell("monoclinic", monoclinic, one, (5, 5, 5)),
            "triclinic": _supercell("triclinic", triclinic, one, (5, 5, 5))}


SYSTEMS = _systems()


@pytest.fixture(scope="module")
def references():
    return {}


def _reference(references, name):
    if name not in references:
        s = SYSTEMS[name]
        recip = np.linalg.inv(s.cell).T
        assert np.all(1.0 / np.linalg.norm(recip, axis=1) >= 3.0 * R_CUT)       # three search cells each way
        i, _, _ = pair_list(s.cell, s.pos, R_CUT)
        wider = len(pair_list(s.cell, s.pos, R_CUT + 1e-6)[0])
        narrower = len(pair_list(s.cell, s.pos, R_CUT - 1e-6)[0])
        assert narrower == len(i) == wider
        x = np.random.default_rng(8).normal(size=(3, 3 * s.n_atoms))
        references[name] = (len(i), x, Operator(s, "spme", tree_pairs=False)(x))
    return references[name]


@pytest.mark.parametrize("updated", [False, True])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("mixed", 2e-6)])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_atoms_on_faces(mbd, references, name, precision, tol, updated):
    s = SYSTEMS[name]
    n_pairs, x, ref = _reference(references, name)
    if updated:
        g = mbd.MBDSystem.from_workload(s.with_(pos=s.pos + 0.1), precision=precision)
        g.update_positions(s.pos)
    else:
        g = mbd.MBDSystem.from_workload(s, precision=precision)
    assert g.info()["n_pairs"] == n_pairs
    y = g.apply_C(torch.tensor(x, device="cuda")).cpu().numpy()
    close(y, ref, tol)
    g.close()
