"""Host threads with a system handle and a stream each: the launches of one thread
do not depend on the limits on dynamic shared memory that another thread sets for
the same kernel (its tile touches fewer pencils, its clusters stage fewer probes,
its field blocks take fewer atoms).  Every energy equals the one the same
handle gave alone."""
import threading

import pytest
import torch

from workloads.systems import random_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mbd():
    from paper_2307_02278_gb300.build import build
    build()
    import paper_2307_02278_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("mesh,order,probes", [((16, 16, 200), 6, (1, 64)), ((20, 24, 20), 8, (40, 128)),
                                               ((16, 288, 16), 6, (1, 64))])
def test_two_threads(mbd, mesh, order, probes):
    """Spreading and clusters; the streamed field kernel; passes without a compiled length."""
    s = random_system(24, 24.0, 12, mesh=mesh, r_cut=9.0, damp_cut=9.0, spline_order=order)
    systems = []
    for _ in probes:
        g = mbd.MBDSystem.from_workload(s, precision="mixed", stream=torch.cuda.Stream())
        g.set_real_space_method("clusters")
        systems.append(g)
    alone = [g.lanczos_energy(r, 64, 5) for g, r in zip(systems, probes)]
    wrong = [[] for _ in probes]

    def work(k):
        for _ in range(40):
            try:
                e = systems[k].lanczos_energy(probes[k], 64, 5)
                if e != alone[k]:
                    wrong[k].append(e)
            except mbd.MBDError as err:
                wrong[k].append(str(err))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(probes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not any(wrong), (wrong[0][:3], wrong[1][:3])
    for g in systems:
        g.close()
