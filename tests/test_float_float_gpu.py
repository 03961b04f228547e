"""The mixed path's float-float kernels at the ends of their ranges: wavenumbers
so low that the Hankel arguments leave the float-float tables below (2^-16), so
high that they leave them above (32) or that box orders leave FP32's scaled
range, geometries in very small and very large units, the QBX orders at the ends
of the coefficient layout, each layer alone. Against the FP64 oracle within the
mixed tolerance 1e-6 (the sums are FP32 with compensation: a few 1e-7)."""
import os
import subprocess
import sys

import numpy as np
import pytest

from qbx_workloads import discretise_curve, fourier_radial
from qbx_workloads.configs import grid_targets

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1602_05301_gb300", "csrc")


def test_table_is_the_generator_output():
    pytest.importorskip("mpmath")
    r = subprocess.run([sys.executable, os.path.join(CSRC, "gen_hankel_table_ff.py")],
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    assert r.stdout == open(os.path.join(CSRC, "hankel_table_ff.h")).read()


@pytest.mark.gpu
@pytest.mark.parametrize("k,unit,panels,p,layers", [
    (3e-4, 1.0, 200, 8, "DS"), (0.03, 1.0, 64, 12, "D"), (3.0, 1e-9, 48, 16, "DS"),
    (3.0, 1e12, 48, 15, "S"), (6.0, 1.0, 80, 0, "S"), (6.0, 1.0, 80, 1, "D"),
    (25.0, 1.0, 64, 16, "DS"), (60.0, 1.0, 128, 12, "DS"), (140.0, 1.0, 300, 6, "D")])
def test_mixed_against_oracle(oracle, k, unit, panels, p, layers):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05301_gb300 import build as b
    b.build()
    from paper_1602_05301_gb300 import qbx
    curve = fourier_radial(unit * np.array([0.0, 0.1, 0.15]), np.array([0.0, 0.4, 1.0]), unit,
                           (0.3 * unit, -0.2 * unit))
    g = discretise_curve(*curve, panels, 16, k=k / unit)
    rng = np.random.default_rng(int(10 * k) + p)
    sig = rng.standard_normal(g.n) + 1j * rng.standard_normal(g.n)
    on = np.arange(0, g.n, 7)
    grid = unit * grid_targets(24, -3.01, 3.0)
    tgt = np.concatenate([g.node_xy[on], grid])
    node = np.concatenate([on, np.full(len(grid), -1)]).astype(np.int64)
    side = np.where(np.arange(len(tgt)) % 2, 1, -1).astype(np.int8)
    lp = qbx.LayerPotential(g.as_dict(), p, sides=2)
    assoc = lp.build(tgt, node, side, mode=qbx.QBX_FMM, p_fmm=30, n_max=40)
    kw = {}
    if "S" in layers:
        kw.update(sigma_S=sig, cS=1j * max(1.0, k))
    if "D" in layers:
        kw.update(sigma_D=sig, cD=unit)
    u = lp.eval(precision=qbx.QBX_MIXED, **kw)
    lp.close()
    u_ref, _ = oracle.layer_potential(
        g.as_dict(), tgt, p, sigma_S=kw.get("sigma_S"), sigma_D=kw.get("sigma_D"),
        cS=kw.get("cS", 0.0), cD=kw.get("cD", 0.0), sides=2, centre_of_target=assoc)
    for sel in (assoc >= 0, assoc < 0):
        assert np.linalg.norm((u - u_ref)[sel]) < 1e-6 * np.linalg.norm(u_ref[sel])
