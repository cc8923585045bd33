"""An update whose pair count exceeds 31 bits: 50,000 atoms pulled together into a ball
whose diameter is below the cutoff have 2.5e9 pairs.  mbd_update_positions
answers MBD_ERR_INVALID_ARG, as mbd_create_system does, and the kernels queued before
the count was read write nothing outside their buffers: going back gives the
products of before, bit for bit."""
import numpy as np
import pytest
import torch

from workloads.systems import System

pytestmark = pytest.mark.gpu

INVALID_ARG = 1


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


def test_update_beyond_31_bits(mbd):
    rng = np.random.default_rng(4)
    n, edge = 50000, 100.0
    grid = np.stack(np.meshgrid(*[np.arange(37)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    pos = (grid + 0.5) * (edge / 37)
    v = rng.normal(size=(n, 3))
    ball = 0.5 * edge + 4.0 * v / np.linalg.norm(v, axis=1)[:, None] * rng.uniform(size=(n, 1)) ** (1.0 / 3.0)
    assert n * (n - 1) > 2 ** 31
    s = System("ball", np.eye(3) * edge, pos, np.full(n, 5.0), np.full(n, 0.5), np.full(n, 3.2), r_cut=8.2,
               damp_cut=8.2, mesh=(200, 200, 200), spline_order=4)
    g = mbd.MBDSystem.from_workload(s, precision="mixed")
    x = torch.randn(2, 3 * n, dtype=torch.float64, device="cuda")
    y, pairs = g.apply_C(x), g.info()["n_pairs"]
    with pytest.raises(mbd.MBDError) as e:
        g.update_positions(ball)
    assert e.value.code == INVALID_ARG
    with pytest.raises(mbd.MBDError) as e:
        mbd.MBDSystem.from_workload(s.with_(pos=ball), precision="mixed")
    assert e.value.code == INVALID_ARG
    g.update_positions(pos)
    assert g.info()["n_pairs"] == pairs and torch.equal(g.apply_C(x), y)
    g.close()
