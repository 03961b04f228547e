"""A density value that is not finite reaches every target: each sums all sources, in
either precision, on the tensor cores and on the CUDA cores."""
import numpy as np
import pytest

from qbx_workloads import discretise_curve, starfish
from qbx_workloads.configs import grid_targets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("engine", [0, 1, 2])
def test_every_target_is_non_finite(engine, bad):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05301_gb300 import build as b
    b.build()
    from paper_1602_05301_gb300 import qbx
    g = discretise_curve(*starfish(0.25, 5), 160, 8, k=5.0)
    sig = np.exp(1j * np.arange(g.n))
    sig[7] = bad
    lp = qbx.LayerPotential(g.as_dict(), 6, sides=2)
    lp.build(grid_targets(40, -3.0, 3.0), mode=qbx.QBX_FMM, p_fmm=20, n_max=20, m2l_engine=engine)
    assert lp.stats()["v_pairs"] > 0
    for precision in (qbx.QBX_FP64, qbx.QBX_MIXED):
        u = lp.eval(sigma_S=sig, cS=1.0, sigma_D=sig, cD=1j, precision=precision)
        assert not np.isfinite(u).any()
        # and the handle is as before
        ok = lp.eval(sigma_S=np.ones(g.n, complex), cS=1.0, precision=precision)
        assert np.isfinite(ok).all()
    lp.close()
