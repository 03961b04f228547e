"""Device memory kept between handles: plans of changing sizes made and dropped in
turn, by one thread and by several at once, give the results of fresh ones, and
what stays behind on the device is bounded."""
import threading

import numpy as np
import pytest

from qbx_workloads import discretise_curve, starfish

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qbxmod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05301_gb300 import build as b
    b.build()
    from paper_1602_05301_gb300 import qbx
    return qbx


def _potential(qbxmod, panels):
    g = discretise_curve(*starfish(0.25, 5), panels, 12, k=4.0)
    sig = np.cos(np.arange(g.n)) + 1j * np.sin(3.0 * np.arange(g.n))
    lp = qbxmod.LayerPotential(g.as_dict(), 6, sides=2)
    lp.build(g.node_xy, np.arange(g.n), np.ones(g.n, np.int8), mode=qbxmod.QBX_FMM, p_fmm=20,
             n_max=20)
    u = lp.eval(sigma_S=sig, cS=1.0, sigma_D=sig, cD=1j)
    lp.close()
    return u


SIZES = [40, 130, 12, 300, 64, 40, 200, 12]


def test_plans_made_and_dropped(qbxmod):
    import torch
    ref = {m: _potential(qbxmod, m) for m in set(SIZES)}
    for m in SIZES:
        assert np.array_equal(_potential(qbxmod, m), ref[m])
    out = {}

    def work(i):
        out[i] = [_potential(qbxmod, m) for m in SIZES[i:] + SIZES[:i]]

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(4):
        for m, u in zip(SIZES[i:] + SIZES[:i], out[i]):
            assert np.array_equal(u, ref[m])
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for m in range(20, 420, 25):
        _potential(qbxmod, m)
    assert free0 - torch.cuda.mem_get_info()[0] < (256 + 64) << 20
