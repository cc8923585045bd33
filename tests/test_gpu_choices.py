"""The atoms per block of the field kernel where the lanes of an atom do not divide
a warp (9 to 12, 17 to 24 and 33 to 40 probes of the FP32 operator: blocks take
3, 5, 6 or 10 atoms at once) on systems just below whole waves of 64 atoms per
block: what mbd_autotune returns stays within the 64 that
mbd_set_launch_choices accepts, and applying it again changes nothing."""
import numpy as np
import pytest
import torch

from workloads.systems import System

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


def _lattice(n, order):
    """n atoms of a simple cubic lattice of spacing 4 bohr, one neighbour shell."""
    k = int(np.ceil(n ** (1.0 / 3.0)))
    grid = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    return System("lattice", np.eye(3) * 4.0 * k, 4.0 * grid + 1.0, np.full(n, 5.0), np.full(n, 0.5),
                  np.full(n, 3.2), r_cut=4.5, damp_cut=4.5, mesh=(48, 48, 48), spline_order=order)


@pytest.mark.parametrize("blocks_per_sm", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("order", [6, 10])
def test_choices_within_their_limit(mbd, order, blocks_per_sm):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = _lattice(64 * blocks_per_sm * sms - 7, order)
    x = torch.randn(3, 3 * s.n_atoms, dtype=torch.float64, device="cuda")
    g = mbd.MBDSystem.from_workload(s, precision="mixed")
    y = g.apply_C(x)
    for probes in (12, 20, 24, 36):
        c = g.autotune(probes)
        assert 1 <= c["field_atoms_per_block"] <= 64, (probes, c)
        g.set_launch_choices(c)
    assert torch.equal(g.apply_C(x), y)
    g.close()
