"""How much device memory the pool takes and gives back."""
import numpy as np
import pytest

from qbx_workloads import circle, discretise_curve

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


def test_large_buffers_are_not_rounded_up(qbxmod):
    """Plans of 2^25 and 2^25 + 1024 targets (buffers of 128 and 512 MB and one step
    above): 48 bytes per target apart, and at most a granule of 2 MB per buffer."""
    import torch
    g = discretise_curve(*circle(0.01), 2, 4, k=1.0)
    used = []
    for n in (1 << 25, (1 << 25) + 1024):
        tgt = np.full((n, 2), 3.0)
        lp = qbxmod.LayerPotential(g.as_dict(), 2, sides=1)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        lp.build(tgt, mode=qbxmod.QBX_DIRECT)
        used.append(free - torch.cuda.mem_get_info()[0])
        lp.close()
    assert used[0] > (1 << 30)
    assert abs(used[1] - used[0]) < 16 * (2 << 20)


def _direct_plan(qbxmod, n):
    lp = qbxmod.LayerPotential(discretise_curve(*circle(0.01), 2, 4, k=1.0).as_dict(), 2, sides=1)
    lp.build(np.full((n, 2), 3.0), mode=qbxmod.QBX_DIRECT)
    return lp


def test_old_blocks_make_room(qbxmod):
    """Blocks of an earlier plan that fill the pool (240 MB) give way to those of later
    plans (132 MB): a plan like the last one takes no new device memory."""
    import torch
    _direct_plan(qbxmod, 6_000_000).close()
    _direct_plan(qbxmod, 3_300_000).close()
    free = torch.cuda.mem_get_info()[0]
    lp = _direct_plan(qbxmod, 3_300_000)
    assert free - torch.cuda.mem_get_info()[0] < (16 << 20)
    lp.close()


def test_release_memory(qbxmod):
    """What the pool keeps after the last handle (here over 100 MB) can be had back, a
    live handle is not affected, and later plans work."""
    import torch
    kept = _direct_plan(qbxmod, 1000)
    _direct_plan(qbxmod, 3_300_000).close()
    free = torch.cuda.mem_get_info()[0]
    n = qbxmod.qbx_release_memory()
    assert n > (100 << 20) and torch.cuda.mem_get_info()[0] - free >= n // 2
    assert qbxmod.qbx_release_memory() == 0
    sig = np.ones(8, complex)
    u = kept.eval(sigma_S=sig, cS=1.0)
    kept.close()
    lp = _direct_plan(qbxmod, 1000)
    assert np.isfinite(u).all() and np.array_equal(u, lp.eval(sigma_S=sig, cS=1.0))
    lp.close()
